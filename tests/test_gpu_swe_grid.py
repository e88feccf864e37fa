"""The FP32 prediction step on either side of the size from which it takes a thread for every four rows (some five million
rows) and with a ragged end: every entry, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,W", [(777 * 1500 + 1, 777), (2049 * 1700 + 3, 2049), (2047 * 3300 + 2, 2047)])
def test_prediction_step_around_the_border_of_its_grids(n, W):
    hn = require_gpu()
    import torch
    rng = np.random.default_rng(n)
    offs = np.array([[-2, -1, 1, 2], [-2 * W, -W, W, 2 * W], [-1, 0, 1, 2], [-W - 1, -W + 1, W - 1, W + 1]])
    bands = rng.uniform(-1, 1, (4, 4, n)).astype(np.float32)
    u, v, w, s = (rng.uniform(-1, 1, n).astype(np.float32) for _ in range(4))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    hn.hn_swe_predict(offs, [[dev(bands[m, k]) for k in range(4)] for m in range(4)], dev(u), dev(v), dev(w), dev(s), out)
    np.testing.assert_array_equal(out.cpu().numpy(), O.swe_predict(offs, bands, u, v, w, s))
