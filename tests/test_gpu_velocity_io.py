"""GPU check of storing and reading the velocity field in one pass: odd sizes, fields that do not
start on a 16-byte boundary, NaN and Inf at the ends, host and device memory, both storages."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,T", [((2, 2, 2), 1), ((3, 5, 7), 3), ((16, 16, 16), 4), ((33, 20, 29), 5)])
@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("off", [0, 1])
def test_velocity_round_trip(shape, T, storage, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    rng = np.random.default_rng(1)
    v = rng.standard_normal((T, 3) + shape).astype(np.float32)
    want = torch.from_numpy(v).bfloat16().float().numpy() if storage else v
    z = np.zeros(shape, np.float32)
    buf = torch.zeros(v.size + off, device="cuda")
    d = buf[off:].reshape(v.shape)
    p = L.default_params(shape[2], shape[1], shape[0], T=T, storage=storage)
    with L.Lddmm(p, z, z) as ctx:
        for src in (v, torch.from_numpy(v).cuda(), d):
            if src is d:
                d.copy_(torch.from_numpy(v))
            ctx.set_velocity(np.zeros_like(v))
            ctx.set_velocity(src)
            assert np.array_equal(ctx.get_velocity(), want)
            out = torch.zeros(v.size + off, device="cuda")[off:].reshape(v.shape)
            assert np.array_equal(ctx.get_velocity(out).cpu().numpy(), want)
        for at in (0, -1):
            for bad in (np.nan, np.inf, -np.inf):
                w = v.copy()
                w.reshape(-1)[at] = bad
                d.copy_(torch.from_numpy(w))
                for src in (w, d):
                    with pytest.raises(L.LddmmError) as ei:
                        ctx.set_velocity(src)
                    assert ei.value.code == L.LDDMM_ERR_NONFINITE
        ctx.set_velocity(v)                      # and the context stays usable
        assert np.array_equal(ctx.get_velocity(), want)
