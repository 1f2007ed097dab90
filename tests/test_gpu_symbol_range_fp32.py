"""GPU check of the FP32 K where the square of the symbol is no normal number: gamma = 1e-20, so that
(gamma + alpha lambda)^2 = 1e-40 and its reciprocal is past FLT_MAX."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# z transforms by columns of 32 (short z), by the folded pass (z > 72; more than 14592 columns)
@pytest.mark.parametrize("shape", [(6, 8, 12), (80, 6, 8), (75, 5, 7), (4, 121, 122)])
def test_subnormal_symbol(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    Z, Y, X = shape
    z = np.zeros(shape, np.float32)
    f = (1e-30 * np.random.default_rng(7).standard_normal(shape)).astype(np.float32)
    gamma = np.float32(1e-20)
    with L.Lddmm(L.default_params(X, Y, Z, T=1, k_mode=0, alpha=0.0, gamma=gamma), z, z) as ctx:
        assert not ctx.apply_K(z).any()
        got = ctx.apply_K(f)
        ctx.step()                                   # no residual: K b = 0 and v stays 0
        assert not ctx.get_velocity().any()
    ref = f.astype(np.float64) / np.float64(gamma) ** 2
    # the square is rounded to a multiple of 2^-149 (7e-6 of it), K itself is good for 2.5e-6
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1e-5
