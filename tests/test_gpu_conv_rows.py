"""GPU check of the tensor-core convolution where its rows can go wrong: grids down to one voxel,
borders, row tiles that end in the volume, one to three row tiles per block, output channels around
16 and up to 256 (filters staged plane by plane), and repeated calls."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P = lambda t: ctypes.c_void_p(t.data_ptr())

# the activations are split into two bf16 (2^-17 of each value), the sums are FP32
TOL = 1e-5


@pytest.mark.parametrize("B,Ci,Co,n,k", [(1, 16, 16, 1, 3), (3, 16, 5, 2, 3), (1, 32, 17, 7, 3),
                                        (2, 48, 16, 33, 3), (8, 16, 48, 32, 3), (1, 64, 192, 16, 3),
                                        (1, 16, 256, 9, 3), (2, 16, 250, 20, 3),
                                        (2, 32, 3, 19, 1), (1, 16, 256, 12, 1), (5, 16, 32, 40, 3)])
def test_conv_rows(B, Ci, Co, n, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    lib = L.load()
    g = torch.Generator().manual_seed(n + Co)
    x = torch.randn(B, Ci, n, n, n, generator=g).cuda()
    w = (torch.randn(Co, Ci, k ** 3, generator=g) / (Ci * k ** 3) ** 0.5).bfloat16().cuda()
    bias = torch.randn(Co, generator=g).cuda()
    ref = torch.zeros(B, Co, n, n, n, dtype=torch.float64, device="cuda")
    xp = torch.nn.functional.pad(x.double(), (k // 2,) * 6)
    for t in range(k ** 3):
        z, y, q = t // (k * k), t // k % k, t % k
        s = xp[:, :, z:z + n, y:y + n, q:q + n]
        ref += torch.einsum("oc,bczyx->bozyx", w[:, :, t].double(), s)
    ref += bias.double()[None, :, None, None, None]
    y = torch.full((B, Co, n, n, n), float("nan"), device="cuda")
    call = lambda y, relu, acc: lib.lddmm_net_conv3d_fwd(P(x), P(w), P(bias), P(y), B, Ci, Co, n, k, relu, acc, None)  # noqa: E731
    assert call(y, 0, 0) == 0
    y2 = torch.empty_like(y)
    assert call(y2, 0, 0) == 0
    yr = torch.empty_like(y)
    assert call(yr, 1, 0) == 0
    ya = y.clone()
    assert call(ya, 0, 1) == 0
    torch.cuda.synchronize()
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())  # noqa: E731
    assert torch.equal(y, y2)
    assert rel(y, ref) < TOL
    assert torch.equal(yr, y.clamp_min(0))
    assert rel(ya, 2 * ref) < TOL
