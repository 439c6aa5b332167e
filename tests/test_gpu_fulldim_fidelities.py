"""Every fidelity and the mask of the full-dimension path.  On rows that are not 16-byte
aligned a handle of one iteration runs the half-step kernels in place, a handle of more the
on-chip blocks: both must give the same bits, as must blocks of one and of many iterations on
aligned rows.  And the FP64 oracle, within the parity tests' bound on u."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U_TOL = 5e-4
ALPHA = {"l2": 10.0, "l1": 1.5, "seg": 20.0}


def _run(H, W, fid, f, m, K, outer):
    from paper_1901_00682_gb300 import _lib as L
    kw = dict(c1=0.2, c2=0.8) if fid == "seg" else {}
    with L.Solver(L.make_params(H, W, fidelity=fid, alpha=ALPHA[fid], inner_iters=K, path="fulldim", **kw)) as s:
        s.load(torch.from_numpy(f).cuda(), None if m is None else torch.from_numpy(m).cuda())
        s.iterate(outer)
        st = s.get_state()
        s.current_energy()   # reports a wait that ran out
    return st


@pytest.mark.parametrize("fid,masked", [("l2", False), ("l2", True), ("l1", False), ("l1", True), ("seg", False)])
@pytest.mark.parametrize("H,W,K", [(3, 5, 3), (128, 128, 10), (127, 133, 10), (129, 232, 4), (300, 337, 25),
                                   (250, 388, 7)])
def test_blocks_and_half_steps_agree(cuda_lib, H, W, K, fid, masked):
    rng = np.random.default_rng(H + W + K)
    f = rng.random((H, W), dtype=np.float32)
    m = (rng.random((H, W)) < 0.2).astype(np.uint8) if masked else None
    n = 3
    a, b = _run(H, W, fid, f, m, K, n), _run(H, W, fid, f, m, 1, n * K)
    for key in a:
        assert torch.equal(a[key], b[key]), key
    kw = dict(c1=0.2, c2=0.8, tau=1.0) if fid == "seg" else {}
    cp = oracle.cp_run(oracle.Problem(H, W, fidelity=fid, alpha=ALPHA[fid], **kw), f.astype(np.float64), n * K, mask=m)
    assert np.abs(a["u"].cpu().numpy().astype(np.float64) - cp.u).max() <= U_TOL
