"""Pyramid merges at the edges of their tiles (1024 child rows) and of the chained scan's
window (256 tiles), with parents of one to eight children that straddle tiles, against the
oracle: keys and counts equal, centroids within the library's tolerance."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_11084_gb300 import vg
from tests._parity import CENTROID_TOL_M, gpu_counts, gpu_keys, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 7, 1023, 1024, 1025, 2049, 262_143, 262_145, 300_007])
@pytest.mark.parametrize("fill", [0.4, 1.0])
def test_tile_edges(rows, fill):
    # `rows` occupied voxels of a cube in Morton order, a share `fill` of the cells taken
    rng = np.random.Generator(np.random.PCG64(rows))
    m = int(np.ceil(rows / fill))
    code = np.sort(rng.permutation(m)[:rows]).astype(np.uint64)
    ijk = np.zeros((rows, 3), np.int64)
    for b in range(21):
        for a in range(3):
            ijk[:, a] |= ((code >> np.uint64(3 * b + a)) & np.uint64(1)).astype(np.int64) << b
    x = ((ijk + rng.uniform(0.1, 0.9, (rows, 3))) * 0.05).astype(np.float32)
    x = np.concatenate([x, x[::3]])[rng.permutation(rows + len(x[::3]))]
    origin = np.zeros(3, np.float32)
    levels = 4
    pyr = vg.pyramid(torch.from_numpy(x).cuda(), 0.05, levels,
                     torch.zeros(3, device="cuda"))
    ref, _ = oracle.pyramid(x, 0.05, levels, origin)
    for k in range(levels):
        keys, cents, counts = ref[k]
        assert np.array_equal(gpu_keys(pyr[k].keys), keys), k
        assert np.array_equal(gpu_counts(pyr[k].counts), counts), k
        assert np.abs(to_np(pyr[k].centroids).astype(np.float64) - cents).max() <= CENTROID_TOL_M
