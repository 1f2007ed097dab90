"""GPU check of the bit-packed mask morphology (rows that end inside a word, one word, thin grids,
radii up to the largest, empty and full masks, unaligned outputs) and of the histogram matching's
FP32 short cut (values on bin edges, many bins, one value, unaligned images), bit for bit."""
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


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 31), (9, 8, 32), (12, 7, 33), (20, 31, 70),
                                   (1, 40, 129), (36, 36, 36)])
@pytest.mark.parametrize("ro,rc", [(0, 0), (1, 0), (0, 5), (2, 3), (0, 16)])
@pytest.mark.parametrize("fill", [0.0, 0.02, 0.6, 0.97, 1.0])
def test_morphology_words(L, shape, ro, rc, fill):
    from oracle import preprocess as OP
    rng = np.random.default_rng(5)
    img = (rng.random(shape) < fill).astype(np.float32)
    buf = torch.zeros(img.size + 1, dtype=torch.uint8, device="cuda")
    out = buf[1:].reshape(shape)                       # one byte off any alignment
    L.mask_morphology(torch.from_numpy(img).cuda(), 0.5, ro, rc, out=out)
    ref = OP.mask_morphology(img, 0.5, ro, rc)
    assert np.array_equal(out.cpu().numpy(), ref.astype(np.uint8))
    aligned = L.mask_morphology(torch.from_numpy(img).cuda(), 0.5, ro, rc)
    assert torch.equal(aligned, out)


@pytest.mark.parametrize("bins,points", [(1, 0), (7, 2), (32, 8), (1000, 64)])
@pytest.mark.parametrize("kind", ["edges", "same", "wide", "noise"])
@pytest.mark.parametrize("n,off", [(1, 0), (4099, 0), (50001, 1)])
def test_histogram_match_bins(L, bins, points, kind, n, off):
    from oracle import preprocess as OP
    rng = np.random.default_rng(n + bins)
    if kind == "edges":                    # multiples of a bin width, and their neighbours in float
        v = rng.integers(0, bins + 1, n).astype(np.float32) * np.float32(0.1)
        v = np.nextafter(v, rng.choice([-np.inf, np.inf], n).astype(np.float32))
    elif kind == "same":
        v = np.full(n, 0.3, np.float32)
    elif kind == "wide":
        v = (rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-30, 30, n)).astype(np.float32)
    else:
        v = rng.lognormal(0, 1, n).astype(np.float32)
    r = rng.normal(0.5, 0.2, n).astype(np.float32)
    m0, m1 = (rng.random(n) < 0.7).astype(np.float32), (rng.random(n) < 0.5).astype(np.float32)
    m0[0] = m1[0] = 1.0
    dev = lambda a: torch.from_numpy(np.concatenate([np.zeros(off, np.float32), a])).cuda()[off:]  # noqa: E731
    ref = OP.histogram_match(v, m0, r, m1, bins, points).astype(np.float32)
    I0 = dev(v)
    got = L.histogram_match(I0, dev(m0), dev(r), dev(m1), bins=bins, points=points)
    assert np.array_equal(got.cpu().numpy(), ref)
    L.histogram_match(I0, dev(m0), dev(r), dev(m1), out=I0, bins=bins, points=points)   # in place
    assert np.array_equal(I0.cpu().numpy(), ref)
