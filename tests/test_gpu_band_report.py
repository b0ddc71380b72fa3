"""A nonzero outside the matrix, which the chase leaves only where an entry of
the band is not finite, is reported: the update answers BDU_EINTERNAL (the
in-place form, which is gated on the chase's status, with its factors
untouched) instead of returning NaN as if nothing had happened."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2509_02840_gb300 import bdu, inputs as I
from test_gpu_nonfinite import EINTERNAL, _dev, _fresh_handle_agrees, _spoiled

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.nan, 1e300])
@pytest.mark.parametrize("where", [0.0, 0.6, 0.999])
@pytest.mark.parametrize("m,n,r,opts", [
    (3, 3, 1, {}), (33, 32, 1, {}), (64, 90, 2, {}), (700, 300, 1, {}), (290, 290, 1, dict(engine=1)),
    (61, 61, 1, dict(precision=bdu.MIXED)), (600, 560, 1, dict(precision=bdu.MIXED, overlap=True)),
])
def test_reported(m, n, r, opts, where, value):
    Q, d, e, P = I.factorization(m, n, config=0, which=7)
    B, C = _spoiled(m, n, r, where, value)
    F = bdu.Factorization(Q, d, e, P, **opts)
    try:
        with pytest.raises(bdu.BduError) as info:
            F.update_dev(B.data_ptr(), C.data_ptr(), r)
            F.sync()
        assert info.value.code == EINTERNAL
    finally:
        F.close()


@pytest.mark.parametrize("m,n", [(61, 61), (200, 150)])
def test_in_place_is_untouched(m, n):
    parts = I.factorization(m, n, config=0, which=4)
    bufs = [_dev(x) for x in parts]
    b, c = _spoiled(m, n, 1, 0.6, np.nan)
    fn = bdu.load().bdu_update_rank1_noalloc
    fn.argtypes = [ctypes.c_int64] * 2 + [ctypes.c_void_p] * 7
    fn.restype = ctypes.c_int
    code = fn(m, n, *[t.data_ptr() for t in bufs], b.data_ptr(), c.data_ptr(),
              torch.cuda.current_stream().cuda_stream)
    assert code == EINTERNAL
    for t, x in zip(bufs, parts):
        assert np.array_equal(t.cpu().numpy(), x.reshape(-1, order="F"))
    _fresh_handle_agrees()
