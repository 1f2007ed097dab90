"""GPU check of what a context holds after a velocity field was refused (NaN or Inf in it): v = 0 and
the maps of v = 0, from whatever memory the field came and in either storage."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPE, T = (9, 13, 17), 3


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    return L


def _context(L, storage=0):
    rng = np.random.default_rng(5)
    I0, I1, M = (rng.random(SHAPE).astype(np.float32) for _ in range(3))
    p = L.default_params(SHAPE[2], SHAPE[1], SHAPE[0], T=T, storage=storage)
    v = rng.standard_normal((T, 3) + SHAPE).astype(np.float32)
    return L.Lddmm(p, I0, I1, M), v, I0


def _sources(v):
    off = torch.zeros(v.size + 1, device="cuda")[1:].reshape(v.shape)
    return {"host": v, "pinned": torch.from_numpy(v).pin_memory(), "device": torch.from_numpy(v).cuda(),
            "unaligned": off.copy_(torch.from_numpy(v))}


def _holds_zero(L, ctx, I0):
    """The same bits as a context whose v was never set."""
    labels = np.arange(I0.size, dtype=np.uint16).reshape(SHAPE)
    fresh, _, _ = _context(L, ctx.params.storage)
    with fresh:
        for c in (ctx, fresh):
            assert not c.get_velocity().any() and not c.get_field(L.LDDMM_FIELD_U10).any()
            assert not c.get_field(L.LDDMM_FIELD_U01).any()
            assert np.array_equal(c.transfer_labels(labels), labels)
        for direction in (0, 1):
            assert np.array_equal(ctx.warp(I0, direction), fresh.warp(I0, direction))
        assert np.array_equal(ctx.get_field(L.LDDMM_FIELD_J0), fresh.get_field(L.LDDMM_FIELD_J0))
        assert ctx.energy()["reg"] == 0.0


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("where", ["host", "pinned", "device", "unaligned"])
@pytest.mark.parametrize("at", [0, -1])
def test_refused_field(L, storage, where, at):
    ctx, v, I0 = _context(L, storage)
    with ctx:
        ctx.set_velocity(v)
        assert not np.array_equal(ctx.warp(I0), I0)         # maps of v are in place
        bad = v.copy()
        bad.reshape(-1)[at] = np.nan if at else np.inf
        with pytest.raises(L.LddmmError) as ei:
            ctx.set_velocity(_sources(bad)[where])
        assert ei.value.code == L.LDDMM_ERR_NONFINITE
        _holds_zero(L, ctx, I0)


def test_refused_field_of_the_exact_gradient(L):
    ctx, v, I0 = _context(L)
    with ctx:
        ctx.set_velocity(v)
        ctx.warp(I0)
        v[-1, -1, -1, -1, -1] = np.nan
        with pytest.raises(L.LddmmError) as ei:
            ctx.energy_grad(torch.from_numpy(v).cuda(), torch.zeros(v.shape, device="cuda"))
        assert ei.value.code == L.LDDMM_ERR_NONFINITE
        _holds_zero(L, ctx, I0)


def test_refused_start_of_a_geodesic(L):
    ctx, v, I0 = _context(L)
    with ctx:
        ctx.set_velocity(v)
        ctx.warp(I0)
        v0 = v[0].copy()
        v0[1, 2, 3, 4] = np.inf
        with pytest.raises(L.LddmmError) as ei:
            ctx.shoot(v0)
        assert ei.value.code == L.LDDMM_ERR_NONFINITE
        _holds_zero(L, ctx, I0)
