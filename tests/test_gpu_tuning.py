"""A launch shape is what its fields say: the shape that hn_mg_get_tuning or an autotuner returns, set again (on the same
hierarchy or another one), runs the kernels that it ran before, and the file of shapes holds it."""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


def kernels(hn, mg, L, b):
    hn.hn_mg_set_profiling(mg, True)
    x, _, _ = hn.hn_mg_solve(mg, L, b)
    out = {(t["name"], t["level"], t["launches"]) for t in hn.hn_mg_kernel_times(mg)}
    hn.hn_mg_set_profiling(mg, False)
    return x, out


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("L", [5, 7, 10])
def test_a_shape_read_and_set_again_runs_the_same_kernels(hn, L, prec, solver):
    coef, b = I.batch_problem(3, L)
    A = hn.hn_band_create(L, coef)
    mgs = [hn.hn_mg_setup(A, prec=prec, solver=solver) for _ in range(2)]
    hn.hn_band_destroy(A)
    try:
        shape = hn.hn_mg_get_tuning(mgs[0])
        want = kernels(hn, mgs[0], L, b)
        for mg in mgs:
            hn.hn_mg_set_tuning(mg, *shape)
            assert hn.hn_mg_get_tuning(mg) == shape
            x, got = kernels(hn, mg, L, b)
            assert got == want[1]
            np.testing.assert_array_equal(x, want[0])
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("L", [7, 9])
def test_an_autotuned_shape_set_on_another_hierarchy_runs_the_same_kernels(hn, L, prec):
    coef, b = I.batch_problem(4, L)
    A = hn.hn_band_create(L, coef)
    mgs = [hn.hn_mg_setup(A, prec=prec) for _ in range(2)]
    hn.hn_band_destroy(A)
    try:
        best, table = hn.hn_mg_autotune(mgs[0], b, reps=1)
        assert len(table) == 3 * 5 * (min(L, 9) - 1) and table[best] == min(table.values())
        shape = hn.hn_mg_get_tuning(mgs[0])
        assert best == (shape[0], shape[1], shape[6], shape[7])
        hn.hn_mg_set_tuning(mgs[1], *shape)
        assert kernels(hn, mgs[1], L, b)[1] == kernels(hn, mgs[0], L, b)[1]
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)


@pytest.mark.parametrize("prec", [0, 1])
def test_a_batch_autotuner_names_the_form_that_it_keeps(hn, prec):
    levels = [7, 5, 6, 7]
    mgs, bs = [], []
    try:
        for j, L in enumerate(levels):
            coef, b = I.batch_problem(j, L)
            A = hn.hn_band_create(L, coef)
            mgs.append(hn.hn_mg_setup(A, prec=prec))
            hn.hn_band_destroy(A)
            bs.append(b)
        best = hn.hn_mg_autotune_batch(mgs, bs, reps=1)
        for mg in mgs:
            shape = hn.hn_mg_get_tuning(mg)
            assert (shape[0], shape[1], shape[2], shape[6]) == best
            assert shape[7] == (0 if shape[6] else -1)
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)
