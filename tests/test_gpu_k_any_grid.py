"""GPU check of the tensor-core K and its fused update on grids of any size: sizes that are no
multiple of 4, 8 or 16, the largest axes of the pre-split passes (264, 256, 256), thin grids, both
storages, with scratch that holds NaN from an earlier call."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(2, 2, 2), (7, 3, 5), (9, 17, 33), (29, 20, 33), (57, 40, 66), (31, 97, 41), (6, 19, 261),
          (5, 8, 264), (4, 256, 21), (256, 6, 18), (8, 32, 64), (40, 8, 12)]


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    L.load()
    return L


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("k_mode,tol", [(1, 2e-5), (2, 1e-2)])   # the bounds of K elsewhere
def test_update_on_any_grid(L, shape, k_mode, tol):
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import synth
    Z, Y, X = shape
    rng = np.random.default_rng(2)
    I0, I1, M = (rng.random(shape).astype(np.float32) for _ in range(3))
    T, eps = 2, 0.5
    v0 = 0.2 * synth.smooth_velocity(T, shape, 1.0, seed=4)
    h = (1.0, 0.8, 1.25)
    ref = O.lddmm_step(v0.astype(np.float64), I0, I1, M, O.Params(T=T, h=h, epsilon=eps))
    kb = (ref.v_new - v0 + eps * 2.0 * v0) / eps            # K b alone
    p = L.default_params(X, Y, Z, T=T, k_mode=k_mode, hx=h[0], hy=h[1], hz=h[2], epsilon=eps)
    with L.Lddmm(p, I0, I1, M) as ctx:
        bad = np.full(shape, np.nan, np.float32)
        ctx.apply_K(bad)                                    # leaves NaN in K's buffers
        ctx.set_velocity(v0)
        ctx.step()
        got = ctx.get_velocity()
        ctx.set_velocity(v0)
        ctx.step()
        assert np.array_equal(got, ctx.get_velocity())
        f = rng.standard_normal(shape).astype(np.float32)
        kf = ctx.apply_K(f)
    assert np.isfinite(got).all()
    # the body force carries the flow's own error (1e-5); its share of v is what the update adds
    assert _rel((got - v0 + eps * 2.0 * v0) / eps, kb) < tol + 2e-5
    assert _rel(kf, O.apply_K(f, 0.02, 1.0, h)) < tol


@pytest.mark.parametrize("shape", [(9, 17, 33), (29, 20, 33), (31, 97, 41), (6, 19, 261), (8, 32, 64)])
def test_bf16_update_on_any_grid(L, shape):
    """The update of a bf16 field is the fp32 field's update rounded once (half of 2^-8, and FP32
    rounding noise)."""
    from paper_1605_02060_gb300 import synth
    Z, Y, X = shape
    rng = np.random.default_rng(2)
    q = lambda a: torch.from_numpy(np.asarray(a, np.float32)).bfloat16().float().numpy()  # noqa: E731
    I0, I1, M = (q(rng.random(shape)) for _ in range(3))
    T = 2
    v0 = q(0.2 * synth.smooth_velocity(T, shape, 1.0, seed=4))
    out = []
    for storage in (0, 1):
        p = L.default_params(X, Y, Z, T=T, k_mode=1, storage=storage, epsilon=0.5)
        with L.Lddmm(p, I0, I1, M) as ctx:
            ctx.set_velocity(v0)
            ctx.step()
            out.append(ctx.get_velocity())
    assert np.all(np.abs(out[1] - out[0]) <= 2.0 ** -8 * np.abs(out[0]) + 1e-6 * np.abs(out[0]).max())
