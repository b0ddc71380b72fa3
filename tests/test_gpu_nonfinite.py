"""Device buffers are not searched for non-finite values, and finite input may
overflow on the band: such an update gives non-finite results or a status,
its rotation records stay inside the factors, and the library works on: a
fresh handle agrees with the oracle bit for bit."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O
from paper_2509_02840_gb300 import bdu, inputs as I

pytestmark = pytest.mark.gpu

ENOTORTH, EINTERNAL = 5, 8


def _dev(x):
    t = torch.from_numpy(np.ascontiguousarray(x.reshape(-1, order="F"))).cuda()
    torch.cuda.synchronize()
    return t


def _spoiled(m, n, r, where, value):
    B, C = (x.copy() for x in I.dense_update(m, n, 1, config=0, r=r))
    X = B if where < 0.5 else C
    X[int(where * 2 % 1 * X.shape[0]), r - 1] = value
    if value == 1e300:  # finite, but u v^T overflows
        B[0, 0] = C[0, 0] = 1e300
    return _dev(B), _dev(C)


def _finish(call):
    """A status is as good an answer as non-finite results."""
    try:
        call()
    except bdu.BduError as err:
        assert err.code in (ENOTORTH, EINTERNAL), err
        return False
    return True


def _fresh_handle_agrees(m=70, n=50):
    Q, d, e, P = I.factorization(m, n, config=0, which=3)
    B, C = I.dense_update(m, n, 0, config=0)
    with bdu.Factorization(Q, d, e, P) as F:
        F.update(B, C)
        got = F.read()
    for a, b in zip(got, O.update(Q, d, e, P, B, C)[:4]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("value", [np.nan, np.inf, 1e300])
@pytest.mark.parametrize("where", [0.1, 0.6, 0.99])
@pytest.mark.parametrize("m,n,r,opts", [
    (61, 61, 1, {}), (90, 64, 2, {}), (64, 90, 1, {}), (700, 520, 1, {}),
    (61, 61, 1, dict(precision=bdu.MIXED)), (700, 520, 2, dict(precision=bdu.MIXED, nb=5)),
    (600, 560, 1, dict(precision=bdu.MIXED, overlap=True)), (1300, 1100, 1, dict(precision=bdu.MIXED)),
])
def test_one_bad_entry(m, n, r, opts, where, value):
    Q, d, e, P = I.factorization(m, n, config=0, which=2)
    B, C = _spoiled(m, n, r, where, value)
    F = bdu.Factorization(Q, d, e, P, **opts)
    try:
        def call():
            F.update_dev(B.data_ptr(), C.data_ptr(), r)
            F.sync()
        if _finish(call):
            assert not np.all(np.isfinite(F.read()[1]))
    finally:
        F.close()
    _fresh_handle_agrees()


@pytest.mark.parametrize("precision", [bdu.FP64, bdu.MIXED])
def test_in_a_batch(precision):
    sizes = [(61, 61, 1), (90, 64, 2), (300, 280, 1), (1200, 1050, 2)]
    fs, ups = [], []
    for i, (m, n, r) in enumerate(sizes):
        fs.append(bdu.Factorization(*I.factorization(m, n, config=0, which=i), precision=precision))
        ups.append(_spoiled(m, n, r, 0.2 + 0.2 * i, np.nan))
    try:
        bdu.update_batch(fs, [b.data_ptr() for b, _ in ups], [c.data_ptr() for _, c in ups], [s[2] for s in sizes])
        for F in fs:
            if _finish(F.sync):
                assert not np.all(np.isfinite(F.read_bidiagonal()[0]))
    finally:
        for F in fs:
            F.close()
    _fresh_handle_agrees()


@pytest.mark.parametrize("m,n", [(61, 61), (200, 150), (1024, 256)])
def test_in_place(m, n):
    Q, d, e, P = I.factorization(m, n, config=0, which=4)
    bufs = [_dev(x) for x in (Q, d, e, P)]
    b, c = _spoiled(m, n, 1, 0.6, np.nan)
    fn = bdu.load().bdu_update_rank1_noalloc
    fn.argtypes = [ctypes.c_int64] * 2 + [ctypes.c_void_p] * 7
    fn.restype = ctypes.c_int
    code = fn(m, n, *[t.data_ptr() for t in bufs], b.data_ptr(), c.data_ptr(),
              torch.cuda.current_stream().cuda_stream)
    assert code in (0, EINTERNAL)
    _fresh_handle_agrees()


@pytest.mark.parametrize("precision", [bdu.FP64, bdu.MIXED])
def test_in_a_tracking_step(precision):
    m, n, k = 150, 130, 24
    g = np.random.default_rng(6)
    Q1, P1 = (I.householder_orthogonal(x, g)[:, :k].copy(order="F") for x in (m, n))
    b, c = g.standard_normal(m), g.standard_normal(n)
    b[40] = np.nan
    tb, tc = _dev(b), _dev(c)
    T = bdu.ThinTracker(Q1, g.uniform(1, 10, k), g.standard_normal(k - 1), P1, precision=precision)
    try:
        _finish(lambda: T.update_dev(tb.data_ptr(), tc.data_ptr()))
    finally:
        T.close()
    _fresh_handle_agrees()
