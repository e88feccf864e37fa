"""The FP64 vector steps on the finest levels (norms, outer defect, update, the steps of CG): a problem
alone, whose tiles go to the warps in turn or as links of 32 (more than 16,384 tiles, from level 11),
gives the bits that it gives in a batch, where blocks share the tiles of all problems."""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


@pytest.mark.parametrize("prec,solver", [(0, 1), (1, 0), (1, 1), (2, 0)])
@pytest.mark.parametrize("levels", [(3, 7, 5, 10), (11, 4, 11, 6), (9,) * 3 + (2, 11)])
def test_fine_steps_alone_and_in_a_batch(hn, levels, prec, solver):
    mgs, bs = [], []
    try:
        for j, L in enumerate(levels):
            A = hn.hn_band_create_bc(L, I.lognormal_coef(L, 60 + j), 15 if j % 2 else 7)
            mgs.append(hn.hn_mg_setup(A, prec=prec, solver=solver))
            hn.hn_band_destroy(A)
            bs.append(I.rhs_uniform_bc(L, 70 + j, 15 if j % 2 else 7))
        xs, stats, status = hn.hn_mg_solve_batch(mgs, list(levels), bs)
        assert status == hn.HN_OK
        for mg, L, b, x, st in zip(mgs, levels, bs, xs, stats):
            y, su, status = hn.hn_mg_solve(mg, L, b)
            assert status == hn.HN_OK and st["relres"] == su["relres"] and st["cycles"] == su["cycles"]
            np.testing.assert_array_equal(x, y)
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)
