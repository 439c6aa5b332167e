"""The tile-fused reverse pass with TV-L1 and segmentation at every block shape, against
autograd through the FP64 restatement.  Both have kinks that float32 and float64 may decide
differently for single pixels, so the bounds are those of the TV-L1 test of
test_gpu_adjoint.py; a wrong derivative is off by its own size."""
import numpy as np
import pytest

from test_gpu_adjoint import _case, _gpu, _ref, _rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fid,mask_prob", [("l1", 0.2), ("l1", 0.0), ("seg", 0.0)])
@pytest.mark.parametrize("shape,tiles", [
    ((64, 64), (2, 2)), ((61, 67), (2, 3)), ((128, 32), (1, 1)),        # blocks 32 wide
    ((128, 128), (2, 2)), ((124, 101), (2, 2)), ((192, 64), (2, 1)),    # 64 wide
    ((128, 256), (1, 2)), ((127, 215), (1, 2)),                         # 128 wide
])
def test_reverse_pass_of_every_fidelity(cuda_lib, shape, tiles, fid, mask_prob):
    f, g, mask = _case(*shape, fid, mask_prob, seed=shape[0] + shape[1])
    N, K, alpha = 4, 5, 1.0 if fid == "seg" else None
    u, gf, ga = _gpu(f, g, mask, *tiles, N, fid, every=3, alpha=alpha, K=K)
    ur, gfr, gar = _ref(f, g, mask, *tiles, N, fid, alpha=alpha, K=K)
    assert np.abs(u - ur).max() <= 5e-4
    assert gar != 0.0 and _rel(gf, gfr) <= 5e-2
    assert abs(ga - gar) <= 1e-2 * abs(gar)
    if mask is not None:
        assert np.all(gf[mask == 1] == 0.0)
