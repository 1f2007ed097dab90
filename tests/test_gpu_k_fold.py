"""GPU check of the folded FP32 axis transforms: even and odd lengths from 2 up, lengths around the
blocks' 24 to 48 pairs, sizes off every vector width, the update fused into the last pass."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(72, 72, 72), (73, 40, 73), (192, 25, 25), (60, 40, 96), (2, 2, 2), (3, 5, 4), (8, 7, 6), (47, 48, 49), (95, 12, 8), (9, 129, 65), (130, 6, 264),
          (17, 96, 97), (33, 3, 300), (5, 64, 512)]

# six sums of at most 257 FP32 products: 6 x 2^-24 x sqrt(257 / 6) = 2.3e-6
TOL = 2.5e-6


@pytest.mark.parametrize("shape", SHAPES)
def test_fp32_K_and_update(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import lddmm as L
    Z, Y, X = shape
    rng = np.random.default_rng(4)
    h, T, eps = (1.0, 0.8, 1.25), 3, 0.5
    f = rng.standard_normal(shape).astype(np.float32)
    I0, I1, M = (rng.random(shape).astype(np.float32) for _ in range(3))
    v0 = (0.1 * rng.standard_normal((T, 3) + shape)).astype(np.float32)
    rel = lambda a, b: np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b)  # noqa: E731
    out = []
    for storage in (0, 1):
        p = L.default_params(X, Y, Z, T=T, hx=h[0], hy=h[1], hz=h[2], k_mode=0, epsilon=eps, storage=storage)
        with L.Lddmm(p, I0, I1, M) as ctx:
            assert rel(ctx.apply_K(f), O.apply_K(f, 0.02, 1.0, h)) < TOL
            if storage:
                break
            for _ in range(2):
                ctx.set_velocity(v0)
                ctx.step()
                out.append(ctx.get_velocity())
    assert np.array_equal(out[0], out[1])
    ref = O.lddmm_step(v0, I0, I1, M, O.Params(T=T, h=h, epsilon=eps))
    kb = (ref.v_new - v0 + eps * 2.0 * v0) / eps
    assert rel((out[0] - v0 + eps * 2.0 * v0) / eps, kb) < TOL + 2e-5    # and the flow's own 1e-5
