"""GPU check of backtracking after the velocity was replaced: the step starts from the field that was
set, not from the one before the last update."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("how", ["set_velocity", "shoot"])
def test_backtracking_step_starts_from_the_set_field(how):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    from paper_1605_02060_gb300 import synth
    shape, T = (12, 14, 16), 3
    rng = np.random.default_rng(6)
    I0, I1 = (rng.random(shape).astype(np.float32) for _ in range(2))
    v = 2.0 * synth.smooth_velocity(T, shape, 1.0, seed=4).astype(np.float32)
    p = L.default_params(shape[2], shape[1], shape[0], T=T, flags=1)
    out = []
    for steps in (0, 2):
        with L.Lddmm(p, I0, I1) as ctx:
            for _ in range(steps):
                ctx.step()
            ctx.set_velocity(v) if how == "set_velocity" else ctx.shoot(v[0])
            e = ctx.step()
            out.append((ctx.get_velocity(), e["total"]))
    # the same launches on the same fields; E is summed by atomics (FP64)
    assert np.array_equal(out[0][0], out[1][0])
    assert abs(out[0][1] - out[1][1]) <= 1e-9 * out[0][1]
