"""bdu_singular_values on graded bidiagonals, each value relatively: the counts
on minors perturb the entries by a few units in their last place, which moves
every singular value, however small, by at most 2n - 1 times as much
relatively (Demmel and Kahan 1990).  Values far below 2^-60 of the norm take the
count that rescales at every step.  The reference is the count of negative
pivots in 120 decimal digits, on both sides of each value returned."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_2509_02840_gb300 import bdu

pytestmark = pytest.mark.gpu


def _below(b2, x):
    """Number of singular values below x > 0 (b2: the Golub-Kahan matrix's squared entries)."""
    q, count = -x, 1
    for v in b2:
        q = -x - (v / q if q else Decimal("Infinity") if v else 0)
        count += q < 0
    return count - (len(b2) + 1) // 2


@pytest.mark.parametrize("scale", [1.0, 1e40])
@pytest.mark.parametrize("order", ["sorted", "shuffled"])
@pytest.mark.parametrize("n,span", [(2, 30), (5, 12), (9, 30), (24, 25), (40, 60)])
def test_relative_accuracy(n, span, order, scale):
    g = np.random.default_rng(n + span)
    d, e = 10.0 ** (-span * g.random(n)), 10.0 ** (-span * g.random(n - 1)) * g.choice([-1.0, 1.0], n - 1)
    if order == "sorted":
        d = -np.sort(-d)
        e[n // 3] = 0.0  # a split beside tiny entries
    d, e = d * scale, e * scale
    with bdu.Factorization(np.eye(n), d, e, np.eye(n)) as F:
        sv = F.singular_values()
    getcontext().prec = 120
    b2 = [Decimal(float(e[i // 2] if i & 1 else d[i // 2])) ** 2 for i in range(2 * n - 1)]
    tol = Decimal(4 * (2 * n - 1)) * Decimal(2.0 ** -52)
    checked = 0
    for j, s in enumerate(sv):
        if s < 1e-80 * sv[0]:  # (64 cuts of the norm's interval by 33 do not resolve less)
            continue
        assert _below(b2, Decimal(float(s)) * (1 - tol)) <= n - 1 - j, j
        assert _below(b2, Decimal(float(s)) * (1 + tol)) >= n - j, j
        checked += s < 2.0 ** -60 * sv[0]
    assert checked or n < 9  # (the smallest orders hold no value that small)
