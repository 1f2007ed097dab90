"""GPU check of the weight and bias gradients at the edges of their tiles: rows that leave a
remainder, fewer voxels than a tile, one voxel, channel counts around the 2/4/8/16 input and 8/16
output channels of a block, and no bias."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P = lambda t: ctypes.c_void_p(t.data_ptr())

# a sum of K random-sign products in FP32 is off by about 2^-24 sqrt(K / 6) of its size; the longest
# chain here has below 1e4 terms
TOL = 5e-6


@pytest.mark.parametrize("B,Ci,Co,n,k", [(1, 2, 16, 9, 3), (2, 3, 20, 33, 3), (3, 17, 16, 40, 3),
                                        (1, 16, 48, 5, 3), (2, 8, 7, 17, 3), (1, 5, 9, 1, 3),
                                        (2, 1, 1, 2, 3), (1, 33, 65, 8, 3), (8, 16, 8, 16, 3),
                                        (1, 40, 5, 7, 1), (2, 16, 3, 24, 1), (1, 1, 1, 1, 1)])
def test_weight_gradient_at_tile_edges(B, Ci, Co, n, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import surrogate as S
    from paper_1605_02060_gb300 import lddmm as L
    lib = L.load()
    rng = np.random.default_rng(7)
    x = rng.standard_normal((B, Ci, n, n, n)).astype(np.float32)
    dy = rng.standard_normal((B, Co, n, n, n)).astype(np.float32)
    gw, gb = S.conv3d_wgrad(x, dy, k)
    xd, dyd = torch.from_numpy(x).cuda(), torch.from_numpy(dy).cuda()
    need = lib.lddmm_net_conv3d_wgrad_scratch(B, Ci, Co, n, k)
    # the scratch may hold anything, and nothing past its end is written
    sc = torch.full((need + 64,), float("nan"), device="cuda")
    dw = torch.ones((Co, Ci, k ** 3), device="cuda")           # sums are added to what is there
    db = torch.ones(Co, device="cuda")
    assert lib.lddmm_net_conv3d_wgrad(P(xd), P(dyd), P(dw), P(db), P(sc), need, B, Ci, Co, n, k,
                                      None) == 0
    only = torch.zeros_like(dw)
    assert lib.lddmm_net_conv3d_wgrad(P(xd), P(dyd), P(only), None, P(sc), need, B, Ci, Co, n, k,
                                      None) == 0
    torch.cuda.synchronize()
    assert torch.isnan(sc[need:]).all()
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    assert rel(only.cpu().numpy().astype(np.float64), gw.reshape(Co, Ci, -1)) < TOL
    assert rel(dw.cpu().numpy() - 1.0, gw.reshape(Co, Ci, -1)) < 1e-4 + TOL
    assert rel(db.cpu().numpy() - 1.0, gb) < 1e-4 + TOL
