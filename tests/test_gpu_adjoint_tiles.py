"""The tile-fused reverse pass at the shapes where it can go wrong: every block size, with and
without padding, clusters of several sizes, uneven subdomains, a mask, one outer iteration
per segment and several, against autograd through the FP64 restatement (the bound of
test_gpu_adjoint.py, 1e-3)."""
import numpy as np
import pytest

from test_gpu_adjoint import _case, _gpu, _ref, _rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,tiles,mask_prob,every", [
    ((64, 64), (2, 2), 0.0, 2), ((61, 67), (2, 3), 0.0, 3),        # blocks 32 wide
    ((120, 30), (2, 1), 0.2, 1), ((128, 32), (1, 1), 0.0, 4),      # ... and taller than 32
    ((128, 128), (2, 2), 0.0, 2), ((124, 101), (2, 2), 0.0, 5),    # 64 wide
    ((100, 60), (1, 1), 0.2, 2), ((192, 64), (2, 1), 0.0, 2),      # ... and taller than 64
    ((128, 256), (1, 2), 0.0, 2), ((112, 128), (1, 1), 0.0, 2),    # 128 wide, without padding and with 7 CTAs
    ((33, 129), (2, 2), 0.0, 2), ((127, 215), (1, 2), 0.2, 2),
])
def test_reverse_pass_of_every_block_shape(cuda_lib, shape, tiles, mask_prob, every):
    f, g, mask = _case(*shape, "l2", mask_prob, seed=shape[0] + shape[1])
    N, K = 4, 5
    u, gf, ga = _gpu(f, g, mask, *tiles, N, "l2", every=every, K=K)
    ur, gfr, gar = _ref(f, g, mask, *tiles, N, "l2", K=K)
    assert np.abs(u - ur).max() <= 5e-4
    assert _rel(gf, gfr) <= 1e-3
    assert abs(ga - gar) <= 1e-3 * abs(gar)
