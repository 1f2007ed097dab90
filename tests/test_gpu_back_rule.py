"""GPU check of the backward sweep between the grids small enough for one plane a thread and those
whose blocks of eight planes fill the GPU: which kernels a step takes, and its fields in both storages."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _fields(shape, T):
    rng = np.random.default_rng(3)
    grid = np.meshgrid(*(np.linspace(0, 3, n) for n in shape), indexing="ij")
    v = np.stack([np.stack([1.5 * np.sin(grid[(c + t) % 3] + 0.7 * grid[c] + t) for c in range(3)])
                  for t in range(T)])
    I0, I1 = (np.sin(grid[0] + k) * np.cos(grid[1]) + 0.3 * grid[2] for k in (0.0, 0.2))
    # fields that bf16 holds exactly, so that every storage sees the oracle's inputs
    q = lambda a: torch.from_numpy(a.astype(np.float32)).bfloat16().float().numpy()  # noqa: E731
    return q(v), q(I0), q(I1), (rng.random(shape) < 0.8).astype(np.float32)


# (z, y, x): 252 four-plane blocks; 260, 600 and 990; 1008 (504 of eight planes), 1320 and 1450; 1820
# (910 of eight planes: more than the SMs hold)
@pytest.mark.parametrize("shape,one", [((25, 47, 190), True), ((50, 77, 60), False), ((80, 80, 80), False),
                                       ((119, 85, 70), False), ((110, 90, 66), True), ((102, 98, 99), True),
                                       ((114, 80, 132), True), ((109, 97, 141), False)])
def test_one_kernel_where_it_is_the_faster_one(shape, one):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    T = 3
    v, I0, I1, M = _fields(shape, T)
    with L.Lddmm(L.default_params(shape[2], shape[1], shape[0], T=T), I0, I1, M) as ctx:
        ctx.set_velocity(v)
        ctx.profile_start(200)
        ctx.step(want_energy=False)
        n = {k: m for k, (m, _) in ctx.profile_stop().items()}
    # the first backward step starts from the identity and has no terms, the last terms stand alone
    want = (T - 1, 1, 1) if one else (0, T, T)
    assert (n.get("flow_back", 0), n["flow_back_terms"], n["flow_back_disp"]) == want


@pytest.mark.parametrize("shape", [(50, 77, 60), (119, 85, 70), (110, 90, 66)])
@pytest.mark.parametrize("storage", [0, 1])
def test_update_from_the_sweep(shape, storage):
    """A step size at which the body force carries v: what J1 and W got wrong would show in it."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import lddmm as L
    O.set_threads(8)
    T, eps = 2, 0.25
    v, I0, I1, M = _fields(shape, T)
    ref = O.lddmm_step(v, I0, I1, M, O.Params(T=T, epsilon=eps))
    p = L.default_params(shape[2], shape[1], shape[0], T=T, storage=storage, epsilon=eps)
    with L.Lddmm(p, I0, I1, M) as ctx:
        ctx.set_velocity(v)
        ctx.step()
        got = ctx.get_velocity()
    du = ref.v_new - v
    assert np.linalg.norm(du) > 2.0 * 2.0 ** -8 * np.linalg.norm(ref.v_new)   # the update shows
    # the repository's bound for one iteration's update; bf16 adds its rounding (half of 2^-7 of v)
    err = got - ref.v_new
    if storage:
        err = np.sign(err) * np.maximum(np.abs(err) - 2.0 ** -8 * np.abs(ref.v_new), 0.0)
    assert np.linalg.norm(err) < 1e-4 * np.linalg.norm(du)
