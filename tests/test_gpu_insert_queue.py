"""The hash insert's queue of runs (a warp's pieces of 128 points, runs within 32 points, 32
added at a time) and the voxel map's packed sums, against the radix sort
and the oracle: ragged sizes around a piece and a chunk, runs that end at every place of a
thread, cells of many points (every carry), frames of all sizes, clearing and refilling."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_11084_gb300 import synth, vg
from tests._parity import assert_decimation_equal, gpu_counts, gpu_keys, to_np

pytestmark = pytest.mark.gpu


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def same(a, b):
    assert np.array_equal(gpu_keys(a.keys), gpu_keys(b.keys))
    assert np.array_equal(gpu_counts(a.counts), gpu_counts(b.counts))
    assert np.array_equal(to_np(a.centroids).view(np.int32), to_np(b.centroids).view(np.int32))


@pytest.mark.parametrize("n", [1, 3, 4, 5, 127, 128, 129, 1023, 1024, 1025, 4099, 200_003])
def test_ragged_sizes(n):
    x = synth.random_cloud(n, seed=n, extent=1.0, nan_frac=0.1, inf_frac=0.02)
    x = np.repeat(x, np.arange(n) % 7 + 1, axis=0)[:n]  # runs of 1 to 7 equal cells
    got = vg.downsample(cuda(x), 0.05, method="hash")
    assert_decimation_equal(got, oracle.downsample(x, 0.05), check_p2v=False)
    same(got, vg.downsample(cuda(x), 0.05, method="sort_lsd"))


@pytest.mark.parametrize("method", ["hash", "auto"])
@pytest.mark.parametrize("posed", [False, True])
def test_runs_of_every_length(method, posed):
    # runs of 1 to 97 points, some of them invalid, from every place of a lane and across
    # lanes, groups of 32 points, warps and chunks; frames that start off a 16-byte boundary
    sizes = [1, 30_002, 129, 50_001, 3]
    x = synth.random_cloud(8_000, seed=9, extent=1.0, nan_frac=0.1)
    x = np.repeat(x, np.arange(len(x)) * 13 % 97 + 1, axis=0)[: sum(sizes)]
    offs = [0] + [int(v) for v in np.cumsum(sizes)]
    kw = {"poses": synth.sensor_poses(len(sizes), seed=2)[0]} if posed else {}
    for p2v in (False, True):
        a = vg.downsample_frames((cuda(x), offs), [0.05] * 5, method=method, point_to_voxel=p2v, **kw)
        b = vg.downsample_frames((cuda(x), offs), [0.05] * 5, method="sort_lsd", point_to_voxel=p2v,
                                 **kw)
        assert a.offsets == b.offsets
        same(a, b)
        assert not p2v or torch.equal(a.point_to_voxel, b.point_to_voxel)


@pytest.mark.parametrize("bits", [9, 10, 11, 14, 20])
def test_index_widths(bits):
    # indices on both sides of 2^10, where the interleave takes a second part
    r = np.random.Generator(np.random.PCG64(bits))
    idx = (r.random((20_000, 3)) * 2 ** bits).astype(np.int64)
    idx[:4] = [[2 ** bits - 1, 0, 0], [0, 2 ** bits - 1, 0], [0, 0, 2 ** bits - 1], [0, 0, 0]]
    x = cuda(((idx + 0.5) * 0.0009765625).astype(np.float32))
    o = torch.zeros(3, device="cuda")
    a = vg.downsample(x, 0.0009765625, o, method="hash")
    ref = oracle.downsample(to_np(x), np.float32(0.0009765625), np.zeros(3, np.float32))
    assert np.array_equal(gpu_keys(a.keys), ref.keys)
    same(a, vg.downsample(x, 0.0009765625, o, method="sort_lsd"))


def test_map_of_crowded_cells_cleared_and_refilled():
    r = np.random.Generator(np.random.PCG64(3))
    m = vg.VoxelMap(50_000, (0.0, 0.0, 0.0), 1.0)
    for turn in range(3):
        n = 400_000 // (turn + 1)
        x = np.concatenate([np.full((n, 3), 0.9999), r.random((20_000, 3)) * 20]).astype(np.float32)
        x = x[r.permutation(len(x))]
        cut = [0, 1, 130, 70_000, len(x)]
        for a, b in zip(cut, cut[1:]):
            m.insert(cuda(x[a:b]))
        got = m.extract()
        same(got, vg.downsample(cuda(x), 1.0, torch.zeros(3, device="cuda"), method="sort_lsd"))
        assert int(gpu_counts(got.counts).max()) >= n
        m.clear()
        assert m.extract().keys.numel() == 0
    m.close()
