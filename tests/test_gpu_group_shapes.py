"""Batches and servers give the bits of the solves alone, whatever launch shape their engine takes: the shape depends
on the number of problems, the largest level, the precision and the options (whole cycles in the cluster tail, one
launch per step, marching sweeps over the one-block tail), and so do the sizes of its launches.  Levels around the
borders of the rule, each on every side of them; Dirichlet and free sides mixed, so that the sweeps of levels 6..8
meet both forms of the restriction."""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu
STEPS = (5, 16, 2, 0, 1, 0, 0, 0)      # one launch per step above the fused tail
MASKS = (15, 10, 7, 15, 1)
WAIT_NS = 120_000_000_000


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


def problem(j, L, bc):
    return I.lognormal_coef(L, 900 + j), I.rhs_uniform_bc(L, 300 + j, bc)


@pytest.mark.parametrize("opts", [{}, {"solver": 1}, {"coarse_solver": 1}, {"pre": 1, "post": 1}])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("count,top", [(2, 5), (2, 6), (4, 8), (7, 7), (4, 9), (5, 9), (8, 6), (8, 9), (11, 8), (12, 8), (3, 10),
                                       (31, 7), (32, 7)])
def test_batches_of_every_shape_give_the_bits_of_the_solves_alone(hn, count, top, prec, opts):
    levels = [top if j % 5 == 1 else 2 + (3 * j) % (min(top, 8) - 1) for j in range(count)]
    masks = [MASKS[j % len(MASKS)] for j in range(count)]
    mgs, bs = [], []
    try:
        for j, (L, bc) in enumerate(zip(levels, masks)):
            coef, b = problem(j, L, bc)
            A = hn.hn_band_create_bc(L, coef, bc)
            mgs.append(hn.hn_mg_setup(A, prec=prec, **opts))
            hn.hn_band_destroy(A)
            bs.append(b)
        xs, stats, status = hn.hn_mg_solve_batch(mgs, levels, bs)
        assert status == hn.HN_OK
        for mg, L, b, x, st in zip(mgs, levels, bs, xs, stats):
            hn.hn_mg_set_tuning(mg, *STEPS)
            y, su, _ = hn.hn_mg_solve(mg, L, b)
            np.testing.assert_array_equal(x, y)
            assert (st["cycles"], st["relres"]) == (su["cycles"], su["relres"])
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("slots", [2, 15, 16, 32])
def test_servers_of_every_shape_give_the_bits_of_the_solves_alone(hn, slots, prec, solver):
    levels = [6, 8, 7, 5, 9, 6, 8, 10, 7, 9, 3, 6, 8, 7, 6, 5, 7, 8]
    problems = [problem(j, L, 15) for j, L in enumerate(levels)]
    srv = hn.hn_server_create(8 << 30, slots)
    try:
        tickets = [hn.hn_mg_submit(srv, L, b, coef, prec=prec, solver=solver) for L, (coef, b) in zip(levels, problems)]
        got = [hn.hn_mg_poll(srv, t, L, timeout_ns=WAIT_NS) for t, L in zip(tickets, levels)]
    finally:
        hn.hn_server_destroy(srv)
    for L, (coef, b), (status, x, st) in zip(levels, problems, got):
        assert status == hn.HN_OK
        A = hn.hn_band_create(L, coef)
        mg = hn.hn_mg_setup(A, prec=prec, solver=solver)
        hn.hn_band_destroy(A)
        hn.hn_mg_set_tuning(mg, *STEPS)
        y, su, _ = hn.hn_mg_solve(mg, L, b)
        hn.hn_mg_destroy(mg)
        np.testing.assert_array_equal(x, y)
        assert st["cycles"] == su["cycles"]
