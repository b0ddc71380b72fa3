"""The chase's pipeline of groups (32 chases a group, a 256-row window a
group): sizes around the edges of groups and of the window, the smallest
problems, tall ones whose spike comes first, and ranks whose later columns
fill a chase's four lanes and wrap around them.  FP64, bit-identical to the
oracle; one thread block (which takes every group in turn) gives the same."""
import numpy as np
import pytest

import oracle as O
from paper_2509_02840_gb300 import bdu, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [0, 1])
@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (2, 1, 1), (2, 2, 1), (3, 2, 2), (32, 32, 1), (33, 33, 1), (34, 33, 1),
                                   (34, 34, 2), (65, 65, 1), (66, 64, 6), (97, 96, 1), (130, 66, 9), (257, 255, 1),
                                   (259, 258, 1), (400, 290, 2), (900, 70, 1)])
def test_group_and_window_edges(m, n, r, engine):
    Q, d, e, P = I.factorization(m, n, config=0, which=11 * m + n)
    B, C = I.dense_update(m, n, h=3, config=0, r=r)
    with bdu.Factorization(Q, d, e, P, precision=bdu.FP64, engine=engine, nb=2) as F:
        F.update(B, C)
        got = F.read()
        st = F.stats()
    want = O.update(Q, d, e, P, B, C)
    for name, a, b in zip("QdeP", got, want):
        assert np.array_equal(a, b), name
    assert st["rot_left"] == [want[4]["left"][p] for p in O.PHASES]
    assert st["rot_right"] == [want[4]["right"][p] for p in O.PHASES]


def test_chases_that_find_nothing_to_do():
    """Zero rows of u end chases before they start, between chases that run."""
    m, n = 150, 120
    Q, P = np.eye(m, order="F"), np.eye(n, order="F")
    g = np.random.default_rng(5)
    d, e = g.uniform(1, 10, n), g.standard_normal(n - 1)
    b, c = g.standard_normal(m), g.standard_normal(n)
    b[g.random(m) < 0.6] = 0.0
    c[g.random(n) < 0.6] = 0.0
    with bdu.Factorization(Q, d, e, P, precision=bdu.FP64, nb=2) as F:
        F.update(b, c)
        got = F.read()
    want = O.update(Q, d, e, P, b.reshape(-1, 1), c.reshape(-1, 1))
    for name, x, y in zip("QdeP", got, want):
        assert np.array_equal(x, y), name


def test_one_block_takes_every_group_of_a_large_column():
    """The watchdog bounds the steps of a group, not of the block that runs them all."""
    n = 1700
    Q = np.eye(n, order="F")
    g = np.random.default_rng(8)
    d, e = g.uniform(1, 10, n), g.standard_normal(n - 1)
    b, c = g.standard_normal(n), g.standard_normal(n)
    got = []
    for engine in (0, 1):
        with bdu.Factorization(Q, d, e, Q, precision=bdu.MIXED, engine=engine) as F:
            F.update(b, c)
            got.append(F.read())
    for name, x, y in zip("QdeP", *got):
        assert np.array_equal(x, y), name
