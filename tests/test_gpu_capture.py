"""Reductions and the defect with norm in a captured graph, reductions on several streams and threads at
once: each call's scratch is its own."""
import threading

import numpy as np
import pytest

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hn():
    return require_gpu()


@pytest.mark.parametrize("n", [1, 16385, 1_000_003])
def test_reductions_captured_and_side_by_side(hn, n):
    import torch
    x = torch.arange(n, device="cuda", dtype=torch.float64) % 7 - 3       # whole numbers: every order gives the same sum
    want = float((x * x).sum())
    out = torch.zeros(2, 2, device="cuda", dtype=torch.float64)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        hn.hn_dot(x, x, out[0, :1], stream)
        hn.hn_nrm2(x, out[1, :1], stream)
    for _ in range(3):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert float(out[0, 0]) == want and float(out[1, 0]) == np.sqrt(want)
    A = hn.hn_band_create(6)
    try:
        b = torch.ones(hn.hn_band_nodes(A), device="cuda", dtype=torch.float64)
        r, norm, again = torch.zeros_like(b), out.new_zeros(1), out.new_zeros(1)
        hn.hn_band_defect_norm_static(A, x.new_zeros(b.numel()), b, r, norm)
        graph = torch.cuda.CUDAGraph()
        zeros = torch.zeros_like(b)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            hn.hn_band_defect_norm_static(A, zeros, b, r, again, stream)
        graph.replay()
        torch.cuda.synchronize()
        assert float(norm) == float(again) == np.sqrt(b.numel()) and torch.equal(r, b)      # x = 0: r = b
    finally:
        hn.hn_band_destroy(A)
    got = {}

    def work(k):
        s = torch.cuda.Stream()
        res = torch.zeros(20, 2, device="cuda", dtype=torch.float64)
        s.wait_stream(torch.cuda.current_stream())
        for i in range(20):
            hn.hn_dot(x, x, res[i, :1], s)
        s.synchronize()
        got[k] = res[:, 0].cpu().numpy()
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(got) == 4 and all((g == want).all() for g in got.values())
