"""The FP64 rotation apply's items (16 rotations x part of a slab's rows):
orders around the edges of items and of the warps they are dealt to, slabs of
2 to 64 rows with a short last one, and the spike, bit-identical to the
oracle whatever the rows per block."""
import numpy as np
import pytest

import oracle as O
from paper_2509_02840_gb300 import bdu, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [0, 2, 6, 8, 64])
@pytest.mark.parametrize("m,n", [(2, 2), (31, 31), (33, 32), (66, 34), (129, 128), (260, 259), (700, 40)])
def test_items_and_slabs(m, n, nb):
    if nb * m * 8 > 227 * 1024:
        pytest.skip("a slab of nb rows does not fit in shared memory: the update refuses nb, as documented")
    Q, d, e, P = I.factorization(m, n, config=0, which=13 * m + n)
    B, C = I.dense_update(m, n, h=1, config=0)
    with bdu.Factorization(Q, d, e, P, precision=bdu.FP64, nb=nb) as F:
        F.update(B, C)
        got = F.read()
    want = O.update(Q, d, e, P, B, C)
    for name, a, b in zip("QdeP", got, want):
        assert np.array_equal(a, b), name
