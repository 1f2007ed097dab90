"""GPU check of the backward sweep in one pass a step on both sides of the grid sizes it is taken for
(256 four-plane blocks, 760 eight-plane ones), with both storage types."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# (z, y, x): 210 and 260 four-plane blocks; 756 and 768 eight-plane ones, with ragged ends
@pytest.mark.parametrize("shape", [(9, 17, 33), (25, 39, 190), (50, 77, 60), (107, 67, 180), (122, 60, 192)])
@pytest.mark.parametrize("storage", [0, 1])
def test_step_on_both_sides_of_the_fused_sweep(shape, storage):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import lddmm as L
    Z, Y, X = shape
    O.set_threads(8)
    rng = np.random.default_rng(3)
    T = 3
    grid = np.meshgrid(*(np.linspace(0, 3, n) for n in shape), indexing="ij")
    v0 = np.stack([np.stack([1.5 * np.sin(grid[(c + t) % 3] + 0.7 * grid[c] + t) for c in range(3)])
                   for t in range(T)]).astype(np.float32)
    I0, I1 = ((np.sin(grid[0] + k) * np.cos(grid[1]) + 0.3 * grid[2]).astype(np.float32) for k in (0.0, 0.2))
    M = (rng.random(shape) < 0.8).astype(np.float32)
    if storage:          # fields that bf16 holds exactly, so that the reference sees the same inputs
        bf = lambda a: torch.from_numpy(a).bfloat16().float().numpy()  # noqa: E731
        v0, I0, I1 = bf(v0), bf(I0), bf(I1)
    ref = O.lddmm_step(v0, I0, I1, M, O.Params(T=T))
    p = L.default_params(X, Y, Z, T=T, k_mode=1, storage=storage)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    with L.Lddmm(p, dev(I0), dev(I1), dev(M)) as ctx:
        ctx.set_velocity(dev(v0))
        e = ctx.step()
        v1 = ctx.get_velocity()
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    # the repository's bounds for one iteration
    if not storage:
        assert rel(v1, ref.v_new) < 1e-4
    assert abs(e["reg"] - ref.E_reg) <= 1e-5 * ref.E_reg
    assert abs(e["data"] - ref.E_data) <= 1e-5 * ref.E_data
    assert abs(e["min_det"] - ref.min_det) <= 1e-4
