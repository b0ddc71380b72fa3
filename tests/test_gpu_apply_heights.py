"""Every slab height that the autotuner of the FP64 apply may choose and report
(bdu_stats.apply_variant) can be asked for (bdu_options.nb), odd ones among
them, and gives the oracle's results bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2509_02840_gb300 import bdu, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [2, 4, 5, 7, 9, 11, 13, 63])
@pytest.mark.parametrize("m,n", [(5, 4), (66, 34), (131, 128), (260, 259)])
def test_heights(m, n, nb):
    Q, d, e, P = I.factorization(m, n, config=0, which=m + nb)
    B, C = I.dense_update(m, n, h=2, config=0)
    with bdu.Factorization(Q, d, e, P, precision=bdu.FP64, nb=nb) as F:
        F.update(B, C)
        got = F.read()
    for name, a, b in zip("QdeP", got, O.update(Q, d, e, P, B, C)):
        assert np.array_equal(a, b), name


@pytest.mark.parametrize("n", [150, 449, 600, 1030])
def test_tuned_height_can_be_asked_for(n):
    Q = np.eye(n)
    g = np.random.default_rng(n)
    d, e = g.uniform(1, 10, n), g.standard_normal(n - 1)
    b, c = g.standard_normal(n), g.standard_normal(n)
    with bdu.Factorization(Q, d, e, Q, precision=bdu.FP64) as F:
        F.update(b, c)
        tuned, got = F.stats()["apply_variant"], F.read()
    for nb in set(tuned):
        with bdu.Factorization(Q, d, e, Q, precision=bdu.FP64, nb=nb) as F:
            F.update(b, c)
            for name, x, y in zip("QdeP", got, F.read()):
                assert np.array_equal(x, y), name
