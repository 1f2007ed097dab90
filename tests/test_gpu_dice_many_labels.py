"""GPU check of Dice on label values past the counts in shared memory, neighbouring voxels of different
labels, and labels up to the last; and that neither costs much more than a few small labels do."""
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


def _context(L):
    z = np.zeros((2, 2, 2), np.float32)
    return L.Lddmm(L.default_params(2, 2, 2, T=1), z, z)


@pytest.mark.parametrize("values", [(2047, 2048), (1, 60000, 60001), (5, 2050, 4098, 65535), (40000,), (1023, 1024)])
@pytest.mark.parametrize("n", [5, 8, 250, 4099])
def test_neighbours_of_different_labels(L, values, n):
    from oracle import lddmm as O
    i = np.arange(n)
    rng = np.random.default_rng(n)
    v = np.array(values, np.uint16)
    with _context(L) as ctx:
        for a, b in ((v[i % len(v)], v[i % (len(v) + 1) % len(v)]),
                     (v[rng.integers(0, len(v), n)], v[rng.integers(0, len(v), n)] * (rng.random(n) < 0.7))):
            a, b = a.astype(np.uint16), b.astype(np.uint16)
            # a mean of a few quotients in FP64
            assert abs(ctx.dice(a, b) - O.dice(a, b)) <= 1e-14


def test_every_label(L):
    from oracle import lddmm as O
    rng = np.random.default_rng(1)
    a = rng.permutation(np.arange(200000) % 65536).astype(np.uint16)
    b = np.where(rng.random(a.size) < 0.5, a, rng.integers(0, 65536, a.size)).astype(np.uint16)
    with _context(L) as ctx:
        # 65535 quotients summed in another order than the oracle's
        assert abs(ctx.dice(a, b) - O.dice(a, b)) <= 1e-12
        assert ctx.dice(a, a) == 1.0


def test_many_labels_cost_little(L):
    """In units of maps of 51 labels: all 65536 labels (dividing them in one block: ten times as much)
    and neighbouring voxels of different large labels (an atomic each: a hundred times as much)."""
    def best(ctx, a, b):
        t = []
        for _ in range(15):
            s = time.perf_counter()
            ctx.dice(a, b)
            t.append(time.perf_counter() - s)
        return min(t)
    dev = lambda a: torch.from_numpy(a.astype(np.int16)).cuda()  # noqa: E731
    rng = np.random.default_rng(2)
    with _context(L) as ctx:
        few, all_ = (dev(rng.integers(0, top, 100000)) for top in (51, 65536))
        assert best(ctx, all_, all_) < 4.0 * best(ctx, few, few)
        i = np.arange(1 << 23)
        few, high = dev(i // 64 % 51), (dev(60000 + i % 2), dev(60000 + i % 3))
        assert best(ctx, *high) < 15.0 * best(ctx, few, few)
