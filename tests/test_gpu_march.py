"""The marching sweeps (a level's down and up part as one pass each) against one launch per step: the
same bits.  Levels from the smallest that marches (one 128-column strip), over several strips and
chunks, to a norm of several groups; every precision that marches, mixed boundaries, a given first
iterate (the lagged check in the first cycle), CG, batches of uneven levels and the server."""
import numpy as np
import pytest

from gpu_util import rand_unknowns, require_gpu
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LR = 2 | 8
STEPS = (5, 16, 2, 0, 1, 0, 0, 0)      # one launch per step above the fused tail


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


def setup(hn, L, coef, bc, **opts):
    A = hn.hn_band_create_bc(L, coef, bc)
    try:
        return hn.hn_mg_setup(A, **opts)
    finally:
        hn.hn_band_destroy(A)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("L,bc", [(7, 15), (7, 7), (8, LR), (9, 15), (9, 1), (10, 10), (11, 15)])
def test_marching_sweeps_give_the_bits_of_the_per_step_kernels(hn, L, bc, solver, prec):
    coef, _ = I.batch_problem(L, L)
    b = I.rhs_uniform_bc(L, 5 + L, bc)
    guess = 0.01 * rand_unknowns(L, bc, 3)
    mg = setup(hn, L, coef, bc, prec=prec, solver=solver)
    try:
        got = [hn.hn_mg_solve(mg, L, b), hn.hn_mg_solve(mg, L, b, guess.copy(), True)]
        hn.hn_mg_set_tuning(mg, *STEPS)
        want = [hn.hn_mg_solve(mg, L, b), hn.hn_mg_solve(mg, L, b, guess.copy(), True)]
        for (x, st, status), (y, su, expected) in zip(got, want):
            assert status == expected == hn.HN_OK
            np.testing.assert_array_equal(x, y)
            assert (st["cycles"], st["outer_iters"], st["relres"]) == (su["cycles"], su["outer_iters"], su["relres"])
    finally:
        hn.hn_mg_destroy(mg)


@pytest.mark.parametrize("prec,count", [(1, 5), (2, 12), (1, 40)])
def test_marching_batches_give_the_bits_of_the_solves_alone(hn, prec, count):
    # the blocks of a launch share the strips and chunks of the problems still in the cycle
    levels = [7 + (3 * j) % 4 if j < 8 else 5 + j % 4 for j in range(count)]
    mgs, bs = [], []
    try:
        for j, L in enumerate(levels):
            coef, b = I.batch_problem(j, L)
            mgs.append(setup(hn, L, coef, 15, prec=prec))
            bs.append(b)
        xs, stats, status = hn.hn_mg_solve_batch(mgs, levels, bs)
        assert status == hn.HN_OK
        for mg, L, b, x, st in zip(mgs, levels, bs, xs, stats):
            hn.hn_mg_set_tuning(mg, *STEPS)
            y, su, _ = hn.hn_mg_solve(mg, L, b)
            np.testing.assert_array_equal(x, y)
            assert st["cycles"] == su["cycles"]
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)


def test_host_issued_marching_iterations_give_the_bits_of_the_graph(hn):
    L = 9
    coef, b = I.batch_problem(2, L)
    mg = setup(hn, L, coef, 15, prec=1)
    try:
        x, _, _ = hn.hn_mg_solve(mg, L, b)
        hn.hn_mg_set_profiling(mg, True)
        y, _, _ = hn.hn_mg_solve(mg, L, b)
        names = {t["name"] for t in hn.hn_mg_kernel_times(mg)}
        hn.hn_mg_set_profiling(mg, False)
        np.testing.assert_array_equal(x, y)
        assert {"sweep_down", "sweep_up", "tail"} <= names and not {"jacobi", "defect", "prolong"} & names, names
    finally:
        hn.hn_mg_destroy(mg)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("L,coarse_L,bc", [(2, 2, 15), (3, 2, 1), (3, 3, LR), (4, 3, 15), (5, 2, LR), (5, 4, 7), (6, 4, 15),
                                           (7, 2, 5)])
def test_one_block_tail_gives_the_bits_of_the_cluster_tail(hn, L, coarse_L, bc, prec):
    # a finest level inside the tail (with its lagged checks) or above it, each coarsest level
    coef, _ = I.batch_problem(L, L)
    b = I.rhs_uniform_bc(L, 9 + L, bc)
    guess = 0.01 * rand_unknowns(L, bc, 4)
    mg = setup(hn, L, coef, bc, prec=prec, coarse_L=coarse_L)
    try:
        got = [hn.hn_mg_solve(mg, L, b), hn.hn_mg_solve(mg, L, b, guess.copy(), True)]
        hn.hn_mg_set_tuning(mg, *STEPS)
        want = [hn.hn_mg_solve(mg, L, b), hn.hn_mg_solve(mg, L, b, guess.copy(), True)]
        for (x, st, status), (y, su, expected) in zip(got, want):
            assert status == expected == hn.HN_OK
            np.testing.assert_array_equal(x, y)
            assert (st["cycles"], st["relres"]) == (su["cycles"], su["relres"])
    finally:
        hn.hn_mg_destroy(mg)
