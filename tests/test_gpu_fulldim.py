"""The full-dimension path on overlapping on-chip blocks: image sides on both sides of the
block edges, several launches per outer iteration, every fidelity.  The steps are constant,
so an outer iteration of K inner ones is K outer iterations of one inner one: launches of K
iterations (wide overlap, few blocks) and of single ones (other blocks) must give the same
bits.  Also against the FP64 oracle, and against a run split at an odd outer iteration and
resumed from exported state (the iterate then lies in the other set of arrays)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U_TOL = 5e-4   # the parity tests' bound on u


def _solver(L, H, W, fid, K):
    kw = dict(c1=0.2, c2=0.8) if fid == "seg" else {}
    return L.Solver(L.make_params(H, W, fidelity=fid, alpha={"l2": 10.0, "l1": 1.5, "seg": 20.0}[fid],
                                  inner_iters=K, path="fulldim", **kw))


@pytest.mark.parametrize("H,W,K", [(1, 1, 3), (127, 128, 10), (128, 129, 10), (129, 232, 10), (233, 131, 10),
                                   (300, 337, 25), (140, 700, 7)])
def test_iterations_per_launch_do_not_change_the_result(cuda_lib, H, W, K):
    from paper_1901_00682_gb300 import _lib as L
    n = 4
    f, _ = synth.rof_image(H, W, 6, 0.05, H + W)
    st = []
    for k, outer in ((K, n), (1, n * K)):
        with _solver(L, H, W, "l2", k) as s:
            s.load(torch.from_numpy(f).cuda())
            s.iterate(outer)
            st.append(s.get_state())
            s.current_energy()   # reports a wait that ran out
    for key in st[0]:
        assert torch.equal(st[0][key], st[1][key]), key
    cp = oracle.cp_run(oracle.Problem(H, W, fidelity="l2", alpha=10.0), f.astype(np.float64), n * K)
    assert np.abs(st[0]["u"].cpu().numpy().astype(np.float64) - cp.u).max() <= U_TOL


@pytest.mark.parametrize("fid,mask", [("l2", True), ("l1", True), ("seg", False)])
@pytest.mark.parametrize("K", [10, 15])
def test_resume_from_either_set(cuda_lib, fid, mask, K):
    from paper_1901_00682_gb300 import _lib as L
    H, W = 250, 301
    rng = np.random.default_rng(3)
    f = torch.from_numpy(rng.random((H, W), dtype=np.float32)).cuda()
    m = torch.from_numpy((rng.random((H, W)) < 0.2).astype(np.uint8)).cuda() if mask else None
    with _solver(L, H, W, fid, K) as s, _solver(L, H, W, fid, K) as t:
        s.load(f, m)
        s.iterate(9)
        whole = s.get_state()
        s.load(f, m)
        s.iterate(3)
        half = s.get_state()
        torch.cuda.synchronize()   # the two handles work on streams of their own
        t.load(f, m)
        t.set_state(half, 3)
        t.iterate(1)
        t.iterate(5)
        parts = t.get_state()
        torch.cuda.synchronize()
    for k in whole:
        assert torch.equal(whole[k], parts[k]), k
