"""FP64 values as FP32 by their bit layout (a hierarchy's bands), to nearest and ties to even like numpy's conversion,
over ordinary, tiny, denormal, overflowing and tied values."""
import numpy as np
import pytest

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -126, 2.0 ** -140, 2.0 ** 126])
def test_bands_round_to_nearest(scale):
    hn = require_gpu()
    L, n = 5, 33
    r = np.random.RandomState(7)
    coef = scale * 2.0 ** r.uniform(-1, 1, (n - 1, n - 1))
    coef[::3, ::2] = scale * (1 + 2.0 ** -24 * r.randint(0, 9, coef[::3, ::2].shape))       # near and on ties
    A = hn.hn_band_create(L, coef.reshape(-1))
    try:
        want = hn.hn_band_get(A)
        mg = hn.hn_mg_setup(A, prec=1)
        try:
            got = hn.hn_mg_get_inner_bands(mg, L, 1)
            got = got[0] if isinstance(got, tuple) else got
        finally:
            hn.hn_mg_destroy(mg)
    finally:
        hn.hn_band_destroy(A)
    with np.errstate(over="ignore"):
        want = want.astype(np.float32)
    np.testing.assert_array_equal(got.view(np.uint32), want.view(np.uint32))
