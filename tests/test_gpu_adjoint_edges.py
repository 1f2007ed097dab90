"""GPU check of the reverse step and of L(L v) where their launches can go wrong: the smallest grids,
rows of whole and broken vectors, axes around a tile, masks that leave part of the volume without a
gradient, rough fields and displacements that leave the grid."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# FP32 sums in any order: a voxel of g takes about 8 terms per step and its gradient 24 products of
# them, 2^-24 each; L L v cancels by (gamma + 12 alpha)^2 / gamma^2 < 3 at alpha = 0.05.  Sampling at
# FP32 coordinates (up to 2^-18 of a voxel at 70) moves an image gradient of order one by as much.
TOL = 1e-4


@pytest.mark.parametrize("rough", [0.0, 3.0])
@pytest.mark.parametrize("flags", [0, 2])
@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 2, 4), (9, 17, 33), (70, 34, 68), (34, 70, 131)])
def test_gradient_at_tile_edges_matches_oracle(shape, flags, rough):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import lddmm as L
    rng = np.random.default_rng(4)
    Z, Y, X = shape
    T = 3
    gz, gy, gx = np.meshgrid(*[np.arange(n) / max(n - 1, 1) for n in shape], indexing="ij")
    I0 = (np.sin(3 * gx + 2 * gy) + np.cos(2 * gz - gx)).astype(np.float32)
    I1 = (np.sin(3 * gx + 2 * gy + 0.3) + np.cos(2 * gz)).astype(np.float32)
    M = ((0.5 + 0.5 * rng.random(shape)) * (gx + gy > 0.4)).astype(np.float32)
    v = np.stack([[np.sin(2 * gx + j + c) + np.cos(3 * gy + gz) for c in range(3)] for j in range(T)])
    v = (v + rough * rng.standard_normal(v.shape)).astype(np.float32)
    h = (1.0, 1.1, 0.9)
    p = L.default_params(X, Y, Z, T=T, sigma=0.5, alpha=0.05, hx=h[0], hy=h[1], hz=h[2], flags=flags)
    Eo, go = O.energy_grad_exact(v, I0, I1, M, O.Params(T=T, sigma=0.5, alpha=0.05, h=h))
    with L.Lddmm(p, I0, I1, M) as ctx:
        E, g = ctx.energy_grad(v)
        E2, g2 = ctx.energy_grad(v)
    assert abs(E - Eo) <= 1e-5 * abs(Eo)
    assert _rel(g, go) < TOL and _rel(g2, go) < TOL
