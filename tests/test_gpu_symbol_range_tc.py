"""GPU check of the tensor-core K where the square of the symbol, or its reciprocal, is no normal
number: (gamma + alpha lambda)^2 = 1e-40 and 1.44e38, on rows of whole vectors and others."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape", [(6, 8, 12), (6, 7, 9), (29, 20, 33)])
@pytest.mark.parametrize("k_mode,tol", [(1, 2e-5), (2, 1e-2)])           # the bounds of K elsewhere
@pytest.mark.parametrize("gamma,scale", [(1e-20, 1e-30), (1.2e19, 1e30)])
def test_symbol_past_the_normal_numbers(shape, k_mode, tol, gamma, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    Z, Y, X = shape
    z = np.zeros(shape, np.float32)
    f = (scale * np.random.default_rng(7).standard_normal(shape)).astype(np.float32)
    gamma = np.float32(gamma)
    with L.Lddmm(L.default_params(X, Y, Z, T=1, k_mode=k_mode, alpha=0.0, gamma=gamma), z, z) as ctx:
        assert not ctx.apply_K(z).any()
        got = ctx.apply_K(f)
        ctx.step()                                   # no residual: K b = 0 and v stays 0
        assert not ctx.get_velocity().any()
    ref = f.astype(np.float64) / np.float64(gamma) ** 2
    # a subnormal square is rounded to a multiple of 2^-149 (7e-6 of 1e-40)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < tol + 1e-5
