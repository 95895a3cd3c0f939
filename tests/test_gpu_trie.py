"""The occupancy trie (AUTO): keys, counts, order, frame offsets,
point_to_voxel and origins equal to the oracle's, and every output bit for bit that of the
global radix sort ("sort_lsd"), over the forms the route accepts: key widths from one level
to six, ragged sizes, runs across warps, cells of many points (carries of the packed sums),
uneven and empty frames, poses, attributes, minimum counts, short outputs and workspaces."""
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
    for x, y in ((a.point_to_voxel, b.point_to_voxel), (a.attrs, b.attrs)):
        assert (x is None) == (y is None)
        if x is not None:
            assert torch.equal(x, y)


def check(x, leaf, origin=None):
    org = None if origin is None else cuda(origin)
    got = vg.downsample(cuda(x), leaf, org, point_to_voxel=True)
    ref = oracle.downsample(x, leaf, origin)
    if len(ref.keys) and np.abs(ref.centroids).max() < 64.0:
        assert_decimation_equal(got, ref)
    else:  # (the library states its centroid bound for coordinates below 64 m)
        assert np.array_equal(gpu_keys(got.keys), ref.keys)
        assert np.array_equal(gpu_counts(got.counts), ref.counts)
        assert np.array_equal(to_np(got.point_to_voxel), ref.point_to_voxel)
    same(got, vg.downsample(cuda(x), leaf, org, method="sort_lsd", point_to_voxel=True))
    plain = vg.downsample(cuda(x), leaf, org)
    same(plain, vg.downsample(cuda(x), leaf, org, method="sort_lsd"))
    return got


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 1023, 1024, 1025, 65_537, 200_003])
def test_ragged_sizes(n):
    check(synth.random_cloud(n, seed=n, extent=2.0, nan_frac=0.05, inf_frac=0.01), 0.02)


@pytest.mark.parametrize("bits", [0, 1, 2, 7, 8, 9, 10, 11, 13, 14, 16, 18, 20, 21])
def test_key_widths(bits):
    # cells per axis up to 2^bits: keys of up to 63 bits, one to six levels
    r = np.random.Generator(np.random.PCG64(bits))
    n = 30_000
    idx = (r.random((n, 3)) * 2 ** bits).astype(np.int64)
    idx[: n // 2] = idx[r.integers(0, 64, n // 2)]  # many points in a few cells
    idx[0] = 2 ** bits - 1
    idx[1] = 0
    # dyadic leaf and coordinates: the indices are exact at every width
    x = ((idx + 0.25 * r.integers(0, 4, (n, 3))) * 0.015625).astype(np.float32)
    check(x, 0.015625, np.zeros(3, np.float32))


@pytest.mark.parametrize("n", [(1 << 21) + 1, 5 << 19, (5 << 19) + 1, (1 << 22) - 1, 1 << 22,
                               (1 << 22) + 1])
def test_threshold_of_the_route(n):
    # shuffled: keys of 26 and 29 bits (either side of what the kernel takes between the
    # sizes), and of more than 32
    x = cuda(synth.fused_map(n, seed=3, extent=(20.0, 20.0, 5.0)))
    for leaf in (0.1, 0.05, 0.008):
        same(vg.downsample(x, leaf), vg.downsample(x, leaf, method="sort_lsd"))


def test_cells_of_many_points():
    # 300,000 points of one cell at its far corner, 3,000 at another's: every carry occurs
    r = np.random.Generator(np.random.PCG64(5))
    x = np.concatenate([np.full((300_000, 3), 0.9999), 1.0 + r.random((3_000, 3)),
                        r.random((5_000, 3)) * 8]).astype(np.float32)
    got = check(x[r.permutation(len(x))], 1.0, np.zeros(3, np.float32))
    assert int(gpu_counts(got.counts).max()) >= 300_000


def test_empty_and_invalid_clouds():
    for x in (np.zeros((0, 3), np.float32), np.full((5000, 3), np.nan, np.float32)):
        got = vg.downsample(cuda(x), 0.05, point_to_voxel=True)
        assert got.keys.numel() == 0 and bool((got.point_to_voxel == -1).all())


@pytest.mark.parametrize("posed", [False, True])
@pytest.mark.parametrize("channels,min_count", [(0, 1), (1, 1), (3, 2), (4, 3)])
def test_frames(posed, channels, min_count):
    sizes = [0, 1, 4097, 0, 20_000, 1024, 1023, 30_001, 0]
    r = np.random.Generator(np.random.PCG64(channels))
    x = cuda(np.concatenate([synth.random_cloud(n, seed=40 + f, extent=1.5 + f, nan_frac=0.1)
                             for f, n in enumerate(sizes)]))
    offs = [0] + [int(v) for v in np.cumsum(sizes)]
    leaves = [0.02, 0.1, 0.05, 0.1, 0.02, 0.3, 0.05, 0.1, 0.02]
    kw = dict(point_to_voxel=True, min_count=min_count)
    if channels:
        kw["attrs"] = torch.from_numpy(r.integers(0, 256, (offs[-1], channels), np.uint8)).cuda()
    if posed:
        poses, _ = synth.sensor_poses(len(sizes), seed=3)
        kw.update(poses=poses, z_limits=np.tile(np.float32([-2.0, 4.0]), (len(sizes), 1)))
    a = vg.downsample_frames((x, offs), leaves, **kw)
    b = vg.downsample_frames((x, offs), leaves, method="sort_lsd", **kw)
    assert a.offsets == b.offsets and torch.equal(a.origins, b.origins)
    same(a, b)
    if not posed and not channels:
        for f, n in enumerate(sizes):
            if n:
                ref = oracle.downsample(to_np(x[offs[f]:offs[f + 1]]), np.float32(leaves[f]))
                assert np.array_equal(gpu_keys(a.frame(f).keys), ref.keys)


def test_many_frames():
    # as many frames as a call takes, their ids the top bits of the keys
    sizes = [97 + f % 5 for f in range(vg.MAX_FRAMES)]
    offs = [0] + [int(v) for v in np.cumsum(sizes)]
    x = cuda(synth.random_cloud(offs[-1], seed=2, extent=3.0))
    a = vg.downsample_frames((x, offs), [0.05] * len(sizes))
    b = vg.downsample_frames((x, offs), [0.05] * len(sizes), method="sort_lsd")
    assert a.offsets == b.offsets
    same(a, b)


@pytest.mark.parametrize("frames,w,h,leaf", [(3, 1280, 720, 0.02), (9, 800, 600, 0.01),
                                             (5, 1280, 720, 0.0005)])
def test_large_coherent_and_incoherent_frames(frames, w, h, leaf):
    # above the size every call takes: camera frames (the sample admits them), and at 0.5 mm
    # more cells than the share of points the buffers hold (left to the sort path), with
    # and without the options, and the sort path after a refusal
    x = cuda(np.concatenate([synth.rgbd_frame(w, h, seed=60 + f) for f in range(frames)]))
    n = w * h
    offs = [f * n for f in range(frames + 1)]
    leaves = [leaf * (1 + f % 2) for f in range(frames)]
    rgb = (torch.arange(3 * x.shape[0], device="cuda") * 37 % 256).to(torch.uint8).reshape(-1, 3)
    for kw in ({}, {"point_to_voxel": True}, {"attrs": rgb, "min_count": 2}):
        a = vg.downsample_frames((x, offs), leaves, **kw)
        b = vg.downsample_frames((x, offs), leaves, method="sort_lsd", **kw)
        assert a.offsets == b.offsets and torch.equal(a.origins, b.origins)
        same(a, b)


@pytest.mark.parametrize("p2v", [False, True])
@pytest.mark.parametrize("origin", [None, (-1.0, -1.0, -1.0)])
def test_large_cloud_that_the_sample_refuses(p2v, origin):
    x = cuda(synth.fused_map(2_900_001, seed=5, extent=(20.0, 20.0, 5.0)))
    o = None if origin is None else cuda(origin)
    same(vg.downsample(x, 0.02, o, point_to_voxel=p2v),
         vg.downsample(x, 0.02, o, point_to_voxel=p2v, method="sort_lsd"))
    few = (x * 0.02).contiguous()  # the same shuffle, a few thousand cells: admitted
    same(vg.downsample(few, 0.02, point_to_voxel=p2v),
         vg.downsample(few, 0.02, point_to_voxel=p2v, method="sort_lsd"))


def test_short_output_and_short_workspace():
    x = cuda(synth.rgbd_frame(640, 480, seed=0))
    n = x.shape[0]
    ref = vg.downsample(x, 0.05, method="sort_lsd")
    b = vg.alloc_buffers(n, "cuda")
    vg.downsample_into(x, 0.05, b, origin_from_min=True, cap=100)
    torch.cuda.synchronize()
    assert int(b.error.item()) == vg.Status.CAPACITY
    assert int(b.num_voxels.item()) == ref.keys.numel()
    assert np.array_equal(gpu_keys(b.keys[:100]), gpu_keys(ref.keys[:100]))
    # a workspace that holds the sort path only is accepted as before, one byte less is not
    small = vg.workspace_bytes(n, vg.method_flag("sort_lsd"))
    assert small < b.workspace.numel()
    c = b._replace(workspace=torch.empty(small, dtype=torch.uint8, device="cuda"))
    vg.downsample_into(x, 0.05, c, origin_from_min=True)
    torch.cuda.synchronize()
    v = int(c.num_voxels.item())
    assert int(c.error.item()) == 0 and v == ref.keys.numel()
    assert torch.equal(c.centroids[:v], ref.centroids)
    with pytest.raises(vg.VGError) as e:
        vg.downsample_into(x, 0.05, c._replace(workspace=c.workspace[:-256]),
                           origin_from_min=True)
    assert e.value.status == vg.Status.WORKSPACE


def test_repeated_calls_in_one_workspace():
    # widths of one, two and four levels in turn: nothing of the call before is read
    x = cuda(synth.rgbd_frame(320, 240, seed=8))
    b = vg.alloc_buffers(x.shape[0], "cuda")
    for leaf in (0.05, 0.0005, 0.02, 0.00001, 0.05):
        vg.downsample_into(x, leaf, b, origin_from_min=True)
        torch.cuda.synchronize()
        assert int(b.error.item()) == 0
        ref = vg.downsample(x, leaf, method="sort_lsd")
        v = int(b.num_voxels.item())
        assert v == ref.keys.numel() and torch.equal(b.keys[:v], ref.keys)
        assert torch.equal(b.centroids[:v], ref.centroids)
