"""The network's pooling, upsampling, channel copies and ReLU backward at the edges of their launch
rules: grids smaller than a block, tensors off the vector alignment, channel counts past a thread's share."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _off(x, k):
    """x on the GPU, k floats past an aligned address."""
    buf = torch.empty(x.numel() + k, device="cuda")
    y = buf[k:].view(x.shape)
    y.copy_(x)
    return y


@pytest.mark.parametrize("off", [0, 1, 2])
@pytest.mark.parametrize("B,C,m,Cy,coff", [(1, 1, 1, 1, 0), (3, 5, 1, 7, 2), (2, 3, 3, 4, 1), (2, 130, 2, 130, 0),
                                           (1, 2, 7, 3, 1), (2, 9, 16, 10, 1)])
def test_resize_copy_and_relu_equal_torch(B, C, m, Cy, coff, off):
    # copies are equal bit for bit; sums of 8 children in FP32 differ by their order: 8 terms of at
    # most 1 in size, so 7 roundings of at most 8 x 2^-24 on either side
    from paper_1605_02060_gb300 import lddmm as L
    lib = L.load()
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    g = torch.Generator().manual_seed(5)
    n, tol = 2 * m, 2 * 7 * 8 * 2.0 ** -24
    fine = _off(torch.rand((B, Cy, n, n, n), generator=g) * 2 - 1, off)
    part = _off(fine[:, coff:coff + C], off)
    coarse = _off(torch.rand((B, C, m, m, m), generator=g) * 2 - 1, off)
    rep = coarse.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)
    eight = torch.nn.functional.avg_pool3d(part, 2) * 8

    y = _off(torch.full((B, Cy, n, n, n), 7.0), off)
    assert lib.lddmm_net_up2(_p(coarse), _p(y), B, C, m, Cy, coff, 0, s) == 0
    assert torch.equal(y[:, coff:coff + C], rep)
    assert bool((y[:, :coff] == 7).all()) and bool((y[:, coff + C:] == 7).all())
    dx = _off(torch.zeros((B, C, m, m, m)), off)
    assert lib.lddmm_net_up2(_p(fine), _p(dx), B, C, m, Cy, coff, 1, s) == 0
    assert float((dx - eight).abs().max()) <= tol

    assert lib.lddmm_net_pool2(_p(part), _p(dx), B * C, n, 0, s) == 0
    assert float((dx - eight / 8).abs().max()) <= tol / 8
    z = _off(torch.zeros((B, C, n, n, n)), off)
    assert lib.lddmm_net_pool2(_p(coarse), _p(z), B * C, n, 1, s) == 0
    assert torch.equal(z, rep * 0.125)

    for nv in (n ** 3, m ** 3):
        src = fine.reshape(-1)[:B * Cy * nv].view(B, Cy, nv)
        d = _off(torch.full((B, C + 1, nv), 3.0), off)
        assert lib.lddmm_net_copy_channels(_p(src), _p(d), B, C, nv, Cy, coff, C + 1, 1, 0, s) == 0
        assert torch.equal(d[:, 1:], src[:, coff:coff + C]) and bool((d[:, 0] == 3).all())
        e = d.clone()
        assert lib.lddmm_net_copy_channels(_p(src), _p(d), B, C, nv, Cy, coff, C + 1, 1, 1, s) == 0
        assert torch.equal(d[:, 1:], e[:, 1:] + src[:, coff:coff + C]) and bool((d[:, 0] == 3).all())

    count = part.numel() - (1 if part.numel() > 5 else 0)
    gr = _off(torch.rand(part.shape, generator=g), off)
    ref = gr.clone()
    ref.view(-1)[:count][part.view(-1)[:count] <= 0] = 0
    assert lib.lddmm_net_relu_bwd(_p(gr), _p(part), count, s) == 0
    assert torch.equal(gr, ref)
