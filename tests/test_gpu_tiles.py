"""The micro-tile kernel of arbitrary subdomain shapes against the plain path, bit for
bit: every block size it chooses, subdomains that fill their block and that are padded by
one row or column or by many, partitions with uneven subdomains, clusters of every size,
sides on the image boundary, interface strips that start off a 16-byte boundary, and inner
counts on both sides of its shared coefficient table.  Both paths evaluate the same float32
operations in the same order, so equality is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ALPHA = {"l2": 10.0, "l1": 1.5, "seg": 20.0}


def _state(L, H, W, NR, NC, fid, mask, K, n, path):
    kw = dict(c1=0.2, c2=0.8) if fid == "seg" else {}
    rng = np.random.default_rng(7 * H + W)
    f = torch.from_numpy(rng.random((H, W), dtype=np.float32)).cuda()
    m = torch.from_numpy((rng.random((H, W)) < 0.2).astype(np.uint8)).cuda() if mask else None
    with L.Solver(L.make_params(H, W, NR, NC, fidelity=fid, alpha=ALPHA[fid], inner_iters=K, path=path, **kw)) as s:
        s.load(f, m)
        s.iterate(n)
        st = s.get_state()
        torch.cuda.synchronize()
        s.current_energy()   # reports a wait that ran out
    return st


@pytest.mark.parametrize("H,W,NR,NC", [
    (32, 32, 1, 1), (31, 33, 1, 1), (96, 96, 3, 3), (95, 97, 3, 3),          # blocks 32 wide
    (65, 32, 1, 1), (128, 96, 1, 4), (250, 61, 2, 2),                        # ... and taller than 32
    (64, 64, 1, 1), (128, 192, 2, 3), (127, 129, 2, 2), (63, 65, 1, 2), (20, 120, 1, 2),   # 64 wide
    (96, 64, 1, 1), (128, 128, 1, 2), (254, 127, 2, 2),                      # ... and taller than 64
    (112, 128, 1, 1), (113, 127, 1, 1), (127, 256, 1, 2), (240, 384, 2, 3),  # 128 wide, clusters of 7 and 8
    (16, 128, 1, 1), (17, 128, 1, 1), (33, 255, 1, 2), (321, 481, 3, 4),     # clusters of 1, 2, 3 and 7
    (139, 60, 2, 2), (281, 148, 5, 10), (241, 292, 10, 4),                   # strips off a 16-byte boundary
])
def test_tile_kernel_equals_plain_path(cuda_lib, H, W, NR, NC):
    from paper_1901_00682_gb300 import _lib as L
    for fid, mask, K in (("l2", False, 7), ("l1", True, 10), ("seg", False, 2), ("l2", True, 65)):
        a, b = (_state(L, H, W, NR, NC, fid, mask, K, 3, path) for path in ("fused", "plain"))
        for k in a:
            assert torch.equal(a[k], b[k]), (fid, mask, K, k)


@pytest.mark.parametrize("path", ["fused", "fulldim"])
def test_loads_share_the_captured_loop(cuda_lib, path):
    """The captured outer loop outlives a load: other data, and a mask that comes, changes
    and goes, give what a new handle gives."""
    from paper_1901_00682_gb300 import _lib as L
    H, W, n = 200, 140, 9
    rng = np.random.default_rng(5)
    grid = (2, 2) if path == "fused" else (1, 1)
    p = dict(sub_rows=grid[0], sub_cols=grid[1], alpha=8.0, inner_iters=6, path=path)
    loads = [(torch.from_numpy(rng.random((H, W), dtype=np.float32)).cuda(),
              torch.from_numpy((rng.random((H, W)) < 0.3).astype(np.uint8)).cuda() if m else None)
             for m in (False, False, True, True, False)]
    with L.Solver(L.make_params(H, W, **p)) as kept:
        for f, m in loads:
            kept.load(f, m)
            kept.iterate(n)
            with L.Solver(L.make_params(H, W, **p)) as new:
                new.load(f, m)
                new.iterate(n)
                a, b = kept.get_state(), new.get_state()
                torch.cuda.synchronize()
            for k in a:
                assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("n,K,fid,mask", [
    (1280, 1, "l2", False), (1280, 2, "seg", False), (1280, 2, "l1", True),      # state in L2
    (2560, 1, "l1", True), (2560, 3, "l2", True), (2560, 4, "l2", False), (2560, 5, "seg", False)])
def test_launches_of_several_waves_equal_plain_path(cuda_lib, n, K, fid, mask):
    """128 x 128 subdomains on both sides of the lines between the persistent and the
    micro-tile kernel."""
    from paper_1901_00682_gb300 import _lib as L
    a, b = (_state(L, n, n, n // 128, n // 128, fid, mask, K, 3, path) for path in ("fused", "plain"))
    for k in a:
        assert torch.equal(a[k], b[k]), k
