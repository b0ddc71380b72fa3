"""The chase's waits between groups run out: failure injection withholds the
first group's progress word (altogether, or only that the group is done); the
warps that wait for it give up after a few thousand polls, the kernel returns
with its status set, and the handle answers BDU_ETIMEOUT.  And a tall update of
high rank, whose spike and steps carry many later columns, does not run out."""
import numpy as np
import pytest

import oracle as O
from paper_2509_02840_gb300 import bdu, inputs as I

pytestmark = pytest.mark.gpu

ETIMEOUT, EPOISONED = 4, 7


@pytest.mark.parametrize("precision,overlap", [(bdu.FP64, False), (bdu.MIXED, True)])
@pytest.mark.parametrize("engine", [0, 1])
@pytest.mark.parametrize("site", [bdu.INJECT_CHASE_STALL, bdu.INJECT_CHASE_UNDONE])
def test_waits_between_groups_expire(site, engine, precision, overlap):
    m, n = 300, 260
    Q, d, e, P = I.factorization(m, n, config=0, which=6)
    B, C = I.dense_update(m, n, 0, config=0)
    F = bdu.Factorization(Q, d, e, P, precision=precision, overlap=overlap, engine=engine, graphs=False)
    try:
        bdu.set_fault_injection(site, 20000)
        try:
            with pytest.raises(bdu.BduError) as info:
                F.update(B, C)
                F.sync()
        finally:
            bdu.set_fault_injection(bdu.INJECT_NONE)
        assert info.value.code == ETIMEOUT
        with pytest.raises(bdu.BduError) as again:
            F.update(B, C)
        assert again.value.code == EPOISONED
    finally:
        F.close()
    with bdu.Factorization(Q, d, e, P) as F:
        F.update(B, C)
        got = F.read()
    for a, b in zip(got, O.update(Q, d, e, P, B, C)[:4]):
        assert np.array_equal(a, b)


def test_tall_update_of_high_rank():
    m, n, r = 1500, 8, 160
    Q, d, e, P = I.factorization(m, n, config=0, which=5)
    B, C = I.dense_update(m, n, 0, config=0, r=r)
    with bdu.Factorization(Q, d, e, P, nb=2) as F:
        F.update(B, C)
        got = F.read()
    for a, b in zip(got, O.update(Q, d, e, P, B, C)[:4]):
        assert np.array_equal(a, b)
