"""Outer iterations in a caller's CUDA graph: every replay advances the iterate, and the handle
goes on from there, bit for bit as without a graph."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path,H,W,grid,K,n_outer", [
    ("fulldim", 250, 301, (1, 1), 10, 1), ("fulldim", 129, 232, (1, 1), 15, 1), ("fulldim", 140, 128, (1, 1), 7, 3),
    ("fulldim", 200, 131, (1, 1), 1, 3), ("fused", 256, 256, (2, 2), 10, 2), ("fused", 1280, 1408, (10, 11), 10, 2)])
def test_replays_advance_the_iterate(cuda_lib, path, H, W, grid, K, n_outer):
    from paper_1901_00682_gb300 import _lib as L
    f = torch.from_numpy(np.random.default_rng(H + W).random((H, W), dtype=np.float32)).cuda()
    p = L.make_params(H, W, *grid, path=path, inner_iters=K)
    with L.Solver(p) as s, L.Solver(p) as t:
        for x in (s, t):
            x.load(f)
            x.iterate(3)
        u, graph = torch.empty_like(f), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            s.set_stream(torch.cuda.current_stream())
            s.iterate(n_outer)
            s.get_u(u)
        s.set_stream(torch.cuda.current_stream())
        for _ in range(3):
            graph.replay()
            t.iterate(n_outer)
            assert torch.equal(u, t.get_u(torch.empty_like(f)))
        if path == "fulldim":   # (the fused path's strips go by the number of iterations the handle counts)
            s.iterate(6)
            t.iterate(6)
            a, b = s.get_state(), t.get_state()
            for k in a:
                assert torch.equal(a[k], b[k]), k
