"""Local solves in several waves, where the multiplier update is a launch of its own and
launches overlap: subdomains that fill their block and that do not, of every block size,
against the plain path bit for bit, over enough outer iterations for the captured loop.  And
the adaptive stop in its kernels for many subdomains against the cluster-barrier kernel."""
import numpy as np
import pytest

from test_gpu_tiles import _state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,NR,NC", [
    (1000, 1500, 34, 50), (1280, 1024, 40, 32),   # blocks 32 wide
    (1600, 960, 16, 32), (1280, 1024, 10, 32),    # ... and taller than 32
    (1100, 1300, 18, 22), (1280, 1280, 20, 20),   # 64 wide
    (1600, 960, 16, 16), (1280, 1024, 10, 16),    # ... and taller than 64
    (1080, 1920, 9, 15), (1280, 1410, 10, 12), (1280, 1408, 10, 11),   # 128 wide
])
@pytest.mark.parametrize("fid,mask,K", [("l2", False, 6), ("l2", True, 3), ("l1", True, 5), ("seg", False, 4)])
def test_several_waves_equal_plain_path(cuda_lib, H, W, NR, NC, fid, mask, K):
    from paper_1901_00682_gb300 import _lib as L
    a, b = (_state(L, H, W, NR, NC, fid, mask, K, 9, path) for path in ("fused", "plain"))
    for k in a:
        assert torch.equal(a[k], b[k]), k


def _adaptive(L, H, W, fid, mask, tol, variant):
    kw = dict(c1=0.2, c2=0.8) if fid == "seg" else {}
    rng = np.random.default_rng(H + W)
    f = np.kron(rng.random((H // 32, W // 32)), np.ones((32, 32))) + 0.05 * rng.standard_normal((H, W))
    m = torch.from_numpy((rng.random((H, W)) < 0.2).astype(np.uint8)).cuda() if mask else None
    p = L.make_params(H, W, H // 128, W // 128, fidelity=fid, alpha={"l2": 8.0, "l1": 1.5, "seg": 20.0}[fid],
                      inner_iters=20, inner_tol=tol, variant=variant, **kw)
    counts = []
    with L.Solver(p) as s:
        s.load(torch.from_numpy(f.astype(np.float32)).cuda(), m)
        for n in (1, 1, 6):   # direct launches and the captured loop
            s.iterate(n)
            counts.append(s.inner_counts()[0])
        st = s.get_state()
        s.current_energy()
    return st, np.array(counts)


@pytest.mark.parametrize("H,W,fid,mask,tol", [
    (1280, 1536, "l2", False, 1e-3), (1280, 1536, "l1", True, 3e-3), (1280, 1536, "seg", False, 1e-3),   # micro-tiles
    (2560, 2560, "l2", False, 1e-3), (2560, 2560, "l2", True, 1e-3), (2560, 2560, "seg", False, 1e-3),   # persistent
    (2560, 2560, "l2", False, 1e-5),   # a tighter tolerance: micro-tiles
])
def test_adaptive_stop_of_many_subdomains(cuda_lib, H, W, fid, mask, tol):
    from paper_1901_00682_gb300 import _lib as L
    (a, ca), (b, cb) = (_adaptive(L, H, W, fid, mask, tol, variant) for variant in (0, 3))
    assert np.array_equal(ca, cb)
    assert tol < 1e-4 or ca.min() < 20   # the rule acts
    for k in a:
        assert torch.equal(a[k], b[k]), k
