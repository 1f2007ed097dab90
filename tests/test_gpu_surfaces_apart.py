"""GPU check of the surface distances of surfaces more than two cells apart: one query or a whole cell
of them (several rounds of 64), few cells that may hold the nearest voxel or more than are kept at
once, and what such surfaces cost."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_02060_gb300 import lddmm as L
    L.load()
    return L


def _masks(shape, kind, rng):
    Z, Y, X = shape
    z, y, x = np.meshgrid(*(np.arange(n) for n in shape), indexing="ij")
    A, B = np.zeros(shape, np.uint8), np.zeros(shape, np.uint8)
    ball = (x - X // 2) ** 2 + (y - Y // 2) ** 2 + (z - Z // 2) ** 2
    if kind == "centre":                       # every cell of the sphere as near as every other
        A[Z // 2, Y // 2, X // 2] = 1
        B[(ball >= 34 ** 2) & (ball < 36 ** 2)] = 1
    elif kind == "five":                       # some more queries in a warp than it takes one by one
        A[Z // 2, Y // 2, X // 2 - 2: X // 2 + 3] = 1
        B[ball >= 36 ** 2] = 1
    elif kind == "noise":                      # cells of several hundred queries, and nearer ones
        A[2:12, 2:12, 2:12] = rng.random((10, 10, 10)) < 0.5
        B[ball < 20 ** 2] = rng.random(int((ball < 20 ** 2).sum())) < 0.5
    else:                                      # two faces
        A[:, :, 0] = 1
        B[:, :, -1] = 1
    return A, B


@pytest.mark.parametrize("kind", ["centre", "five", "noise", "faces"])
@pytest.mark.parametrize("shape", [(75, 77, 80)])
@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (0.5, 1.25, 2.0)])
def test_surfaces_apart(L, shape, kind, h):
    from oracle import metrics as OM
    A, B = _masks(shape, kind, np.random.default_rng(3))
    z = np.zeros(shape, np.float32)
    p = L.default_params(shape[2], shape[1], shape[0], hx=h[0], hy=h[1], hz=h[2], T=1)
    with L.Lddmm(p, z, z) as ctx:
        got, back = ctx.surface_distance(A, B), ctx.surface_distance(B, A)
    hd, md = OM.surface_distances(A.astype(bool), B.astype(bool), h)
    assert got[:2] == back[:2] and got[2:] == back[:1:-1]
    # these spacings' squares are short binary fractions: FP32 compares them exactly, and only the
    # FP64 root's rounding is left
    assert abs(got[0] - hd) <= 1e-14 * hd and abs(got[1] - md) <= 1e-14 * md


def test_the_space_between_costs_little(L):
    """264x160x228: two ellipsoids at opposite ends and one voxel in either corner cost a few times the
    same ellipsoid against itself two voxels on (about twice and as much; 30 and 18 times when every
    query walked all cells between)."""
    shape = (228, 160, 264)
    z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in shape), indexing="ij")
    ell = lambda c, dx=0: sum(((q - c * n - s) / (0.18 * n)) ** 2  # noqa: E731
                              for q, n, s in ((x, 264, dx), (y, 160, 0), (z, 228, 0))).lt(1).to(torch.uint8)
    first, last = torch.zeros(shape, dtype=torch.uint8, device="cuda"), torch.zeros(shape, dtype=torch.uint8, device="cuda")
    first[0, 0, 0] = 1
    last[-1, -1, -1] = 1
    zero = torch.zeros(shape, device="cuda")
    with L.Lddmm(L.default_params(264, 160, 228, T=1), zero, zero) as ctx:
        def best(a, b):
            t = []
            for _ in range(9):
                s = time.perf_counter()
                ctx.surface_distance(a, b)
                t.append(time.perf_counter() - s)
            return min(t)
        near = best(ell(0.2), ell(0.2, 2))
        assert best(ell(0.2), ell(0.8)) < 6.0 * near
        assert best(first, last) < 3.0 * near
