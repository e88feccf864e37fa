"""The tails over a cluster of 16 blocks (FP64: levels to 6; FP32 / FP16 alone: to 8; the lagged check and,
for a problem whose finest level is in it, all cycles in one launch) and the FP64 steps on finer levels
against the general kernels: the same bits, for each top level, coarsest level, boundary mask, zero and
given iterates (nonzero on Dirichlet nodes too), CG, a cycle limit and batches."""
import numpy as np
import pytest

from gpu_util import rand_unknowns, require_gpu
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GENERAL = [(5, 16, 2, 0, 1, 0, 0, 0), (6, 8, 0, 0, 0, 0, 0, 1)]


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


def outcome(hn, mg, L, b, guess=None):
    try:
        x, st, status = hn.hn_mg_solve(mg, L, b) if guess is None else hn.hn_mg_solve(mg, L, b, guess.copy(), True)
    except hn.HnError as e:                 # (CG can break down from a residual on Dirichlet nodes)
        return np.zeros(0), {"cycles": 0, "relres": 0.0}, e.status
    return x, st, status


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("prec,L,coarse,bc", [
    (0, 2, 2, 15), (0, 3, 2, 7), (0, 3, 3, 15), (0, 4, 2, 15), (0, 4, 3, 10), (0, 4, 4, 1), (0, 5, 2, 15), (0, 5, 4, 5),
    (0, 5, 3, 8), (0, 6, 2, 15), (0, 6, 3, 4), (0, 6, 4, 2), (0, 6, 2, 1), (0, 7, 2, 15), (0, 8, 3, 11), (0, 9, 2, 6), (0, 10, 2, 15),
    (1, 4, 2, 15), (1, 6, 2, 15), (1, 6, 3, 4), (2, 6, 4, 2), (1, 7, 4, 10), (2, 7, 2, 15), (1, 8, 2, 15), (2, 8, 3, 11),
    (1, 8, 4, 5), (1, 8, 2, 8), (2, 8, 2, 1), (1, 9, 2, 15), (2, 10, 3, 2)])
def test_cluster_tails_give_the_bits_of_the_general_tail(hn, prec, L, coarse, bc, solver):
    A = hn.hn_band_create_bc(L, I.lognormal_coef(L, 31 + L), bc)
    opts = dict(prec=prec, solver=solver, coarse_L=coarse)
    b = I.rhs_uniform_bc(L, 5 + L, bc)
    guess = 0.01 * rand_unknowns(L, bc, 3)
    rim = guess + 0.01                      # nonzero on the Dirichlet nodes
    got = []
    for shape in [None] + GENERAL:
        mg = hn.hn_mg_setup(A, **opts)
        short = hn.hn_mg_setup(A, max_cycles=2, tol=0.0, **opts)
        try:
            if shape:
                for m in (mg, short):
                    hn.hn_mg_set_tuning(m, max(shape[0], coarse), *shape[1:])
            got.append([outcome(hn, mg, L, b), outcome(hn, mg, L, b, guess), outcome(hn, mg, L, b, rim),
                        outcome(hn, short, L, b), outcome(hn, short, L, b, guess)])
        finally:
            hn.hn_mg_destroy(mg)
            hn.hn_mg_destroy(short)
    hn.hn_band_destroy(A)
    for other in got[1:]:
        for (x, st, status), (y, su, expected) in zip(got[0], other):
            assert status == expected
            np.testing.assert_array_equal(x, y)
            assert (st["cycles"], st["relres"]) == (su["cycles"], su["relres"])


@pytest.mark.parametrize("levels", [(6,), (6, 4, 5), (7, 6, 3, 8), (5,) * 12])
def test_wide_tail_in_batches(hn, levels):
    mgs, bs = [], []
    try:
        for j, L in enumerate(levels):
            coef, b = I.batch_problem(j, L)
            A = hn.hn_band_create(L, coef)
            mgs.append(hn.hn_mg_setup(A, prec=0))
            hn.hn_band_destroy(A)
            bs.append(b)
        xs, stats, status = hn.hn_mg_solve_batch(mgs, list(levels), bs)
        assert status == hn.HN_OK
        for mg, L, b, x, st in zip(mgs, levels, bs, xs, stats):
            y, su, status = hn.hn_mg_solve(mg, L, b)
            assert status == hn.HN_OK and st["cycles"] == su["cycles"] and st["relres"] == su["relres"]
            np.testing.assert_array_equal(x, y)
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)
