"""The compact form after a partial run of BHU and of the symmetric variant:
I - Y SL Y^T and I - W SR W^T are the products of the reflectors returned.
BHU leaves the last column of SR after steps <= n - 2 with its diagonal entry
alone, to be completed as bdu.h says (tolerance as for a complete run in
test_gpu_bhu.py: 1e-12 times the order)."""
import numpy as np
import pytest

from oracle import bhu as H
from test_gpu_bhu import _case, run_factor
from test_gpu_tri import _case as _tri_case, run_tri

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,t,rk", [(12, 9, 1, 1), (12, 9, 2, 1), (12, 9, 7, 1), (12, 9, 8, 1), (64, 64, 61, 1),
                                      (64, 64, 62, 1), (64, 64, 63, 1), (300, 200, 57, 3), (530, 529, 300, 8)])
def test_bhu(m, n, t, rk):
    d, e, u, v = _case(m, n, m + 3 * t)
    if rk > 1:
        g = np.random.default_rng(t)
        u, v = g.standard_normal((m, rk)), g.standard_normal((n, rk))
    r = run_factor(m, n, d, e, u, v, steps=t)
    Q, P = H.factors(r["Y"], r["W"], m, n)
    assert np.abs(np.eye(m) - r["Y"] @ r["SL"] @ r["Y"].T - Q).max() <= 1e-12 * m
    SR, W, k = r["SR"], r["W"], r["SR"].shape[0]
    if 1 < k and t <= n - 2:
        assert not np.any(SR[:k - 1, k - 1])
        SR[:k - 1, k - 1] = -2.0 * SR[:k - 1, :k - 1] @ (W[:, :k - 1].T @ W[:, k - 1])
    assert np.abs(np.eye(n) - W @ SR @ W.T - P).max() <= 1e-12 * n


@pytest.mark.parametrize("n,t", [(12, 1), (12, 2), (12, 10), (12, 11), (64, 61), (300, 57), (530, 300)])
def test_tri(n, t):
    a, b, u, rho = _tri_case(n, n + t)
    r = run_tri(n, a, b, u, rho, steps=t)
    Q, _ = H.factors(r["Y"], np.zeros((1, 0)), n, 1)
    assert np.abs(np.eye(n) - r["Y"] @ r["S"] @ r["Y"].T - Q).max() <= 1e-12 * n
