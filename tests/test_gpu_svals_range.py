"""The Sturm counts of bdu_singular_values run on minors that are rescaled every
few steps: magnitudes from 2^-400 to 2^400, exact zeros in runs, and orders
around the rescaling interval, against a library SVD of the scaled matrix."""
import numpy as np
import pytest

import oracle as O
from paper_2509_02840_gb300 import bdu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** -400, 1.0, 2.0 ** 400])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 33, 130])
def test_scales_and_orders(n, scale):
    g = np.random.default_rng(n)
    d, e = g.uniform(1, 10, n), g.standard_normal(n - 1)
    if n > 30:
        d[5:9] = 0.0
        e[4:9] = 0.0
        e[20:24] = 0.0
    with bdu.Factorization(np.eye(n), d * scale, e * scale, np.eye(n)) as F:
        sv = F.singular_values()
    ref = O.singular_values(d, e)
    assert np.max(np.abs(sv / scale - ref)) <= 2e-14 * ref[0]
