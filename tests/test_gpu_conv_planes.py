"""GPU check of the tensor-core convolution's splits: blocks of several planes that end inside the
grid, output channels divided between blocks (with a ragged last part), and a grid so wide that the
filter's planes are staged one at a time."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
P = lambda t: ctypes.c_void_p(t.data_ptr())

# the activations are split into two bf16 (2^-17 of each value), the sums are FP32
TOL = 1e-5


def _ref(x, w, bias, zs):
    n = x.shape[-1]
    xp = torch.nn.functional.pad(x[:, :, max(zs[0] - 1, 0):zs[-1] + 2].double(),
                                 (1, 1, 1, 1, zs[0] == 0, zs[-1] == n - 1))
    m = len(zs)
    ref = bias.double()[None, :, None, None, None].repeat(x.shape[0], 1, m, n, n)
    for t in range(27):
        z, y, q = t // 9, t // 3 % 3, t % 3
        ref += torch.einsum("oc,bczyx->bozyx", w[:, :, t].double(), xp[:, :, z:z + m, y:y + n, q:q + n])
    return ref


@pytest.mark.parametrize("B,Ci,Co,n", [(8, 16, 16, 45), (5, 48, 20, 37), (8, 32, 96, 30), (8, 64, 192, 15),
                                       (1, 64, 200, 8), (3, 128, 128, 5), (1, 32, 33, 65), (1, 16, 3, 500)])
def test_conv_planes(B, Ci, Co, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    lib = L.load()
    g = torch.Generator(device="cuda").manual_seed(n + Co)
    x = torch.randn(B, Ci, n, n, n, generator=g, device="cuda")
    w = (torch.randn(Co, Ci, 27, generator=g, device="cuda") / (27 * Ci) ** 0.5).bfloat16()
    bias = torch.randn(Co, generator=g, device="cuda")
    y = torch.full((B, Co, n, n, n), float("nan"), device="cuda")
    assert lib.lddmm_net_conv3d_fwd(P(x), P(w), P(bias), P(y), B, Ci, Co, n, 3, 0, 0, None) == 0
    torch.cuda.synchronize()
    assert not bool(torch.isnan(y).any())
    for z0 in range(0, n, 16) if n < 100 else (0, 249, n - 2):
        zs = list(range(z0, min(z0 + (16 if n < 100 else 2), n)))
        ref = _ref(x, w, bias, zs)
        assert float((y[:, :, zs[0]:zs[-1] + 1].double() - ref).norm() / ref.norm()) < TOL
