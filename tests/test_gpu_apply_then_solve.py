"""A solve does not depend on what single-kernel calls (hn_mg_apply) left in the hierarchy's vectors: after
calls on every level with vectors that are nonzero everywhere, also on Dirichlet nodes, it gives the bits of a
solve on a fresh hierarchy."""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LR = 2 | 8


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


def outcomes(hn, mgs, levels, bs):
    alone = [hn.hn_mg_solve(mg, L, b) for mg, L, b in zip(mgs, levels, bs)]
    xs, stats, status = hn.hn_mg_solve_batch(mgs, levels, bs)
    assert status == hn.HN_OK
    return [(x, st["cycles"], st["relres"]) for x, st, _ in alone] + [(x, st["cycles"], st["relres"]) for x, st in zip(xs, stats)]


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("bc", [15, LR])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("levels", [(6, 4), (8, 7), (10, 9)])
def test_solves_after_single_kernel_calls_give_the_bits_of_fresh_ones(hn, levels, prec, bc, solver):
    dt = np.float64 if prec == 0 else np.float32
    coefs = [I.batch_problem(80 + L, L)[0] for L in levels]
    bs = [I.rhs_uniform_bc(L, 11 + L, bc) for L in levels]
    mgs = []
    try:
        for L, coef in zip(levels, coefs):
            A = hn.hn_band_create_bc(L, coef, bc)
            mgs += [hn.hn_mg_setup(A, prec=prec, solver=solver) for _ in range(2)]
            hn.hn_band_destroy(A)
        fresh, used = mgs[0::2], mgs[1::2]
        rng = np.random.default_rng(5)
        for mg, L in zip(used, levels):
            def vec(l):
                return rng.uniform(1, 2, ((1 << l) + 1) ** 2).astype(dt)
            for l in range(3, L + 1):
                hn.hn_mg_apply(mg, hn.HN_OP_RESTRICT, l, prec != 0, vec(l))
                hn.hn_mg_apply(mg, hn.HN_OP_PROLONG_ADD, l, prec != 0, vec(l - 1), vec(l))
            for l in range(2, L + 1):
                for op in (hn.HN_OP_SPMV, hn.HN_OP_DEFECT, hn.HN_OP_JACOBI, hn.HN_OP_JACOBI_ZERO):
                    hn.hn_mg_apply(mg, op, l, prec != 0, vec(l), vec(l))
        for got, want in zip(outcomes(hn, used, list(levels), bs), outcomes(hn, fresh, list(levels), bs)):
            np.testing.assert_array_equal(got[0], want[0])
            assert got[1:] == want[1:]
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)
