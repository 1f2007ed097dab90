"""GPU check of the flow kernels on both sides of the block counts at which their marches change
depth (256, 2048 and 8192 four-plane blocks): one step against the oracle, both integrators."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# (z, y, x): 252 and 260 blocks, 2048 and 2128, 7800 and 8208, with ragged ends
@pytest.mark.parametrize("shape", [(25, 47, 190), (50, 77, 60), (128, 128, 128), (75, 108, 255),
                                   (154, 200, 255), (227, 143, 250)])
@pytest.mark.parametrize("rk", [False, True])
def test_step_on_both_sides_of_the_march_depths(shape, rk):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import lddmm as L
    Z, Y, X = shape
    if rk and Z * Y * X > 3e6:
        pytest.skip("the oracle's RK4 takes minutes at this size; the kernels are chosen alike")
    O.set_threads(8)
    rng = np.random.default_rng(3)
    T = 2
    grid = np.meshgrid(*(np.linspace(0, 3, n) for n in shape), indexing="ij")
    v0 = np.stack([np.stack([1.5 * np.sin(grid[(c + t) % 3] + 0.7 * grid[c] + t) for c in range(3)])
                   for t in range(T)]).astype(np.float32)
    I0, I1 = ((np.sin(grid[0] + k) * np.cos(grid[1]) + 0.3 * grid[2]).astype(np.float32) for k in (0.0, 0.2))
    M = (rng.random(shape) < 0.8).astype(np.float32)
    ref = O.lddmm_step(v0, I0, I1, M, O.Params(T=T, integrator="rk4" if rk else "sl"))
    p = L.default_params(X, Y, Z, T=T, k_mode=1, flags=4 if rk else 0)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    with L.Lddmm(p, dev(I0), dev(I1), dev(M)) as ctx:
        ctx.set_velocity(dev(v0))
        e = ctx.step()
        v1 = ctx.get_velocity()
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    # the repository's bounds for one iteration
    assert rel(v1, ref.v_new) < 1e-4 and rel(v1 - v0, ref.v_new - v0) < 1e-4
    assert abs(e["reg"] - ref.E_reg) <= 1e-5 * ref.E_reg
    assert abs(e["data"] - ref.E_data) <= 1e-5 * ref.E_data
    assert abs(e["min_det"] - ref.min_det) <= 1e-4
