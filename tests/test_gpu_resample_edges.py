"""The grid resampling where an axis is one voxel, or shorter or longer than a tile of the kernel."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("src,dst", [((1, 1, 1), (2, 3, 5)), ((1, 6, 5), (4, 1, 300)), ((5, 1, 6), (1, 300, 3)),
                                     ((4, 3, 1), (300, 2, 1)), ((3, 4, 5), (17, 9, 33)), ((40, 30, 20), (1, 1, 1)),
                                     ((6, 5, 4), (16, 257, 1))])
@pytest.mark.parametrize("ncomp", [1, 3])
def test_resample_at_tile_edges_matches_oracle(src, dst, ncomp):
    # 7 nested lerps a + t (b - a) of values at most M with weights rounded once to FP32: below
    # 12 2^-24 M for the operations, 3 2^-25 2 M for the weights, one more rounding for the scale
    from oracle import lddmm as O
    from paper_1605_02060_gb300 import lddmm as L
    rng = np.random.default_rng(6)
    f = rng.standard_normal((2, 3) + src).astype(np.float32)
    sc = (1.5, 0.75, 2.0) if ncomp == 3 else (1.25, 1.0, 1.0)
    got = L.resample(torch.from_numpy(f).cuda(), dst, ncomp=ncomp, scale=sc).cpu().numpy()
    for t in range(2):
        for c in range(3):
            a = f[t, c]
            for ax in range(3):            # the oracle samples between two voxels along every axis
                a = np.repeat(a, 2, ax) if a.shape[ax] == 1 else a
            k = sc[c] if ncomp == 3 else sc[0]
            assert np.abs(got[t, c] - k * O.resample(a, dst)).max() <= 16 * 2.0 ** -24 * np.abs(f).max() * k
