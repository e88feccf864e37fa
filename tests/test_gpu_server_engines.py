"""The server's engines against solves alone, bit for bit: an engine of one slot that was built for a larger
request than the one it runs (its launches for the levels that the request does not have do nothing, but keep
the order of the launches around them)."""
import numpy as np
import pytest

from gpu_util import require_gpu, solve
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu
WAIT_NS = 120_000_000_000


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_one_slot_runs_smaller_requests_on_a_larger_engine(hn, prec, solver):
    levels = [11, 9, 10, 7, 9]
    problems = [I.batch_problem(70 + j, L) for j, L in enumerate(levels)]
    alone = [solve(hn, L, b, coef, prec=prec, solver=solver) for L, (coef, b) in zip(levels, problems)]
    srv = hn.hn_server_create(8 << 30, 1)
    try:
        for _ in range(2):
            tickets = [hn.hn_mg_submit(srv, L, b, coef, prec=prec, solver=solver) for L, (coef, b) in zip(levels, problems)]
            for t, L, (x, st, _) in zip(tickets, levels, alone):
                status, y, su = hn.hn_mg_poll(srv, t, L, timeout_ns=WAIT_NS)
                assert status == hn.HN_OK
                np.testing.assert_array_equal(y, x)
                assert su["cycles"] == st["cycles"]
    finally:
        hn.hn_server_destroy(srv)
