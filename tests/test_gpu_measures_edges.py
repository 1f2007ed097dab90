"""GPU check of the surface distances where the cell search can go wrong (surfaces many cells
apart, grids that end inside a cell, anisotropic spacing, single voxels, odd and even counts) and
of Dice with large labels, ragged lengths and unaligned maps."""
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
    A, B = np.zeros(shape, np.uint8), np.zeros(shape, np.uint8)
    if kind == "corners":                 # the whole box between them
        A[0, 0, 0] = 1
        B[-1, -1, -1] = 1
    elif kind == "far":                   # a blob at one end, scattered voxels at the other
        A[: Z // 4, : Y // 3, : X // 5] = 1
        B[Z - Z // 4:, Y // 2:, X - X // 5:] = rng.random((Z // 4, Y - Y // 2, X // 5)) < 0.3
        B[-1, -1, -1] = 1
    elif kind == "noise":
        A[:] = rng.random(shape) < 0.02
        B[:] = rng.random(shape) < 0.5
        A[0, 0, 0] = 1
    else:                                 # nested boxes, every face a cell or more away
        A[1:-1, 1:-1, 1:-1] = 1
        B[Z // 2: Z // 2 + 1, Y // 3: Y // 2 + 1, X // 3: X // 2 + 1] = 1
    return A, B


@pytest.mark.parametrize("shape", [(2, 2, 2), (8, 16, 24), (9, 17, 33), (41, 23, 70)])
@pytest.mark.parametrize("kind", ["corners", "far", "noise", "nested"])
@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (0.5, 1.25, 2.0)])
def test_surface_distance_cells(L, shape, kind, h):
    from oracle import metrics as OM
    if kind in ("far", "nested") and min(shape) < 8:
        pytest.skip("the pattern needs a larger grid")
    A, B = _masks(shape, kind, np.random.default_rng(3))
    z = np.zeros(shape, np.float32)
    p = L.default_params(shape[2], shape[1], shape[0], hx=h[0], hy=h[1], hz=h[2], T=1)
    with L.Lddmm(p, z, z) as ctx:
        got = ctx.surface_distance(torch.from_numpy(A).cuda(), B)
    hd, md = OM.surface_distances(A.astype(bool), B.astype(bool), h)
    assert got[2] == int(OM.surface(A.astype(bool)).sum())
    assert got[3] == int(OM.surface(B.astype(bool)).sum())
    # these spacings' squares are short binary fractions: FP32 compares them exactly, and only the
    # FP64 root's rounding is left
    assert abs(got[0] - hd) <= 1e-14 * hd and abs(got[1] - md) <= 1e-14 * max(md, 1e-300)


@pytest.mark.parametrize("n,off", [(1, 0), (7, 1), (4096, 0), (100003, 0), (100003, 3)])
@pytest.mark.parametrize("top", [3, 2047, 2048, 65535])
def test_dice_labels(L, n, off, top):
    from oracle import lddmm as O
    rng = np.random.default_rng(n + top)
    runs = rng.integers(1, 40, n)
    a = np.repeat(rng.integers(0, top + 1, n), runs)[:n].astype(np.uint16)
    b = np.where(rng.random(n) < 0.9, a, rng.integers(0, top + 1, n)).astype(np.uint16)
    a[-1] = top
    z = np.zeros((2, 2, 2), np.float32)
    dev = lambda q: torch.from_numpy(np.concatenate([np.zeros(off, np.int16), q.view(np.int16)])).cuda()[off:]  # noqa: E731
    with L.Lddmm(L.default_params(2, 2, 2, T=1), z, z) as ctx:
        got = ctx.dice(dev(a), dev(b))
        assert abs(got - ctx.dice(a, b)) == 0
    assert abs(got - O.dice(a, b)) <= 1e-12
