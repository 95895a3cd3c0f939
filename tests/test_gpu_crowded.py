"""Crowded clouds without order: few cells, or one cell with much of the cloud, points shuffled.
The hash insert merges the queued runs of keys that come back, the occupancy trie sums the rows
that many runs meet in each block first; their rows, and a voxel map's, are the radix sort's
bit for bit."""
import numpy as np
import pytest
import torch

from paper_2102_11084_gb300 import vg
from tests._parity import gpu_counts, gpu_keys, to_np

pytestmark = pytest.mark.gpu
LEAF = 0.0625


def crowd(n, cells, hot=0.0, seed=0):
    """n points in `cells` cells, a share `hot` of them in one; offsets up to the far corner."""
    r = np.random.Generator(np.random.PCG64(seed + n + cells))
    at = r.permutation(64 ** 3)[:cells]
    c = at[r.integers(0, cells, n)]
    c = np.where(r.random(n) < hot, at[0], c)
    ijk = np.stack((c % 64, c // 64 % 64, c // 4096), 1)
    off = np.where(r.random((n, 1)) < 0.5, 0.999, r.random((n, 3)))
    x = ((ijk + off) * LEAF).astype(np.float32)
    x[::101] = np.nan
    return torch.from_numpy(x).cuda()


def same(a, b):
    assert np.array_equal(gpu_keys(a.keys), gpu_keys(b.keys))
    assert np.array_equal(gpu_counts(a.counts), gpu_counts(b.counts))
    assert np.array_equal(to_np(a.centroids).view(np.int32), to_np(b.centroids).view(np.int32))


CLOUDS = [(1, 1, 0.0), (33, 2, 0.0), (4097, 3, 0.0), (200_003, 1, 0.0), (200_003, 2, 0.0),
          (200_003, 10, 0.0), (200_003, 33, 0.0), (200_003, 1000, 0.0), (200_003, 50_000, 0.1),
          (200_003, 50_000, 0.5), (3_000_001, 2, 0.0), (3_000_001, 200_000, 0.3)]


@pytest.mark.parametrize("n,cells,hot", CLOUDS)
def test_hash_and_map(n, cells, hot):
    x = crowd(n, cells, hot)
    o = torch.zeros(3, device="cuda")
    ref = vg.downsample(x, LEAF, o, method="sort_lsd")
    same(vg.downsample(x, LEAF, o, method="hash"), ref)
    m = vg.VoxelMap(max(2 * cells, 64), [0.0, 0.0, 0.0], LEAF)
    cut = n // 3
    for part in (x[:cut], x[cut:]):  # (two inserts, the second into occupied cells)
        if part.shape[0]:
            m.insert(part.contiguous())
    same(m.extract(), ref)


@pytest.mark.parametrize("p2v", [False, True])
@pytest.mark.parametrize("n,cells,hot", CLOUDS + [(131_071, 7, 0.0), (131_072, 7, 0.0),
                                                  (900_001, 4095, 0.0), (900_001, 4096, 0.0),
                                                  (900_001, 4097, 0.0), (2_600_000, 70_000, 0.2)])
def test_auto(n, cells, hot, p2v):
    # rows up to a block's table of them and one more; rows that take an entry once met again
    x = crowd(n, cells, hot)
    o = torch.zeros(3, device="cuda")
    ref = vg.downsample(x, LEAF, o, method="sort_lsd", point_to_voxel=p2v)
    got = vg.downsample(x, LEAF, o, point_to_voxel=p2v)
    same(got, ref)
    if p2v:
        assert torch.equal(got.point_to_voxel, ref.point_to_voxel)


@pytest.mark.parametrize("channels", [1, 2, 3, 4])
@pytest.mark.parametrize("n,cells,hot", [(200_003, 3, 0.0), (900_001, 2049, 0.0),
                                         (900_001, 2048, 0.0), (900_001, 60_000, 0.4)])
def test_auto_attributes(n, cells, hot, channels):
    x = crowd(n, cells, hot)
    r = np.random.Generator(np.random.PCG64(channels))
    at = torch.from_numpy(r.integers(0, 256, (n, channels), np.uint8)).cuda()
    at[: n // 2] = 255
    o = torch.zeros(3, device="cuda")
    ref = vg.downsample(x, LEAF, o, method="sort_lsd", attrs=at)
    got = vg.downsample(x, LEAF, o, attrs=at)
    same(got, ref)
    assert torch.equal(got.attrs, ref.attrs)
