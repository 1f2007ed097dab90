"""GPU check of the map refresh, the warps and the label transfer on both sides of the block count at
which their marches change depth (256 four-plane blocks), with planes and rows left over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("T,rk", [(1, False), (4, False), (3, True)])
@pytest.mark.parametrize("shape", [(2, 2, 2), (9, 17, 33), (25, 47, 190), (51, 77, 61)])
def test_maps_warps_and_labels(shape, T, rk):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import lddmm as L
    Z, Y, X = shape
    grid = np.meshgrid(*(np.linspace(0, 3, n) for n in shape), indexing="ij")
    v = np.stack([np.stack([1.5 * np.sin(grid[(c + t) % 3] + 0.7 * grid[c] + t) for c in range(3)])
                  for t in range(T)]).astype(np.float32)
    img = (np.sin(3 * grid[0]) * np.cos(grid[1]) + 0.3 * grid[2]).astype(np.float32)
    lab = (np.arange(Z * Y * X) % 60000).astype(np.uint16).reshape(shape)
    po = O.Params(T=T, integrator="rk4" if rk else "sl")
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    p = L.default_params(X, Y, Z, T=T, flags=4 if rk else 0)
    with L.Lddmm(p, dev(img), dev(img), dev(np.ones(shape, np.float32))) as ctx:
        ctx.set_velocity(v)
        to = [ctx.warp(img, 0), ctx.warp(img, 1)]
        u = [ctx.get_field(L.LDDMM_FIELD_U10), ctx.get_field(L.LDDMM_FIELD_U01)]
        J0, got = ctx.get_field(L.LDDMM_FIELD_J0), ctx.transfer_labels(lab)
    # nearest neighbour by the float32 rule: the same voxels
    assert np.array_equal(got, O.transfer_labels(lab, u[0]))
    # a lookup rounds its coordinate by 2^-18 of a voxel at 190, 2^-19 at 77, less below, times a slope
    # of at most 0.4 a voxel there (2 on the smallest grid, where it rounds by 2^-23), and makes nine
    # operations of 2^-24 on values below 2
    for d in (0, 1):
        ref = O.warp(img.astype(np.float64), u[d].astype(np.float64))
        assert np.abs(to[d] - ref).max() < 1e-5
    assert np.abs(J0 - to[0]).max() < 2e-6
    # the maps: T lookups of displacements below 8 voxels, of slope below 3 a voxel, 2^-18 each
    g = O._grid(shape)

    def follow(steps, sign):
        w = np.zeros((3,) + shape)
        for j in steps:
            d = O._step_disp(v[j], po, sign, g)
            w = d + O.interp_vec(w, g[2] + d[0], g[1] + d[1], g[0] + d[2])
        return w

    assert np.abs(u[0] - follow(range(T), -1.0)).max() < 1e-4
    assert np.abs(u[1] - follow(range(T - 1, -1, -1), 1.0)).max() < 1e-4
