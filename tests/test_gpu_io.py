"""The kernels that start and end a solve: vectors in device memory give the bits of host arrays, at odd and
ragged sizes and at offsets inside an allocation, beyond the problems of one launch; a rejected right-hand
side leaves the result as it was, a zero one gives zeros whatever the iterate, results that share memory
come out one after the other."""
import numpy as np
import pytest

from gpu_util import rand_unknowns, require_gpu
from paper_0904_4152_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


def setup(hn, L, **opts):
    A = hn.hn_band_create(L)
    try:
        return hn.hn_mg_setup(A, **opts)
    finally:
        hn.hn_band_destroy(A)


@pytest.mark.parametrize("L,prec", [(2, 0), (3, 1), (6, 2), (7, 1), (10, 0), (11, 1)])
def test_device_vectors_give_the_bits_of_host_arrays(hn, L, prec):
    import torch
    b, guess = I.rhs_uniform(L, 9), 0.01 * rand_unknowns(L, 15, 4)
    N = b.size
    mg = setup(hn, L, prec=prec)
    try:
        hold = torch.full((2 * N + 8,), 7.0, dtype=torch.float64, device="cuda")
        db, dx = hold[2:2 + N], hold[N + 3:2 * N + 3]         # both on 16-byte boundaries (N is odd)
        for given in (False, True):
            db.copy_(torch.from_numpy(b))
            dx.copy_(torch.from_numpy(guess))
            x, st, _ = hn.hn_mg_solve(mg, L, b, guess.copy(), given)
            y, su, _ = hn.hn_mg_solve(mg, L, db, dx, given)
            np.testing.assert_array_equal(y.cpu().numpy(), x)
            np.testing.assert_array_equal(db.cpu().numpy(), b)
            assert (st["cycles"], st["relres"]) == (su["cycles"], su["relres"])
            assert all(float(hold[k]) == 7.0 for k in (0, 1, N + 2, 2 * N + 3))
        db.zero_()
        y, st, status = hn.hn_mg_solve(mg, L, db, dx, True)
        assert status == hn.HN_OK and float(y.abs().max()) == 0.0
        db[0] = 1.0                                           # a Dirichlet node
        dx.fill_(3.0)
        with pytest.raises(hn.HnError) as e:
            hn.hn_mg_solve(mg, L, db, dx)
        assert e.value.status == hn.HN_ERR_ARG and float((dx - 3.0).abs().max()) == 0.0
    finally:
        hn.hn_mg_destroy(mg)


@pytest.mark.parametrize("count,shared", [(1, False), (97, False), (3, True)])
def test_batches_of_device_vectors(hn, count, shared):
    import torch
    levels = [4 if shared else 2 + j % 5 for j in range(count)]
    mgs = [setup(hn, L, prec=1) for L in levels]
    try:
        bs = [I.rhs_uniform(L, j) for j, L in enumerate(levels)]
        db = [torch.from_numpy(b).cuda() for b in bs]
        one = torch.zeros(bs[0].size, dtype=torch.float64, device="cuda")
        dx = [one if shared else torch.zeros_like(b) for b in db]
        xs, _, status = hn.hn_mg_solve_batch(mgs, levels, bs)
        ys, _, status_d = hn.hn_mg_solve_batch(mgs, levels, db, dx)
        assert status == status_d == hn.HN_OK
        for j in range(count):
            np.testing.assert_array_equal(ys[j].cpu().numpy(), xs[-1 if shared else j])
    finally:
        for mg in mgs:
            hn.hn_mg_destroy(mg)
