"""The minimum-count filter's chained scan (tiles of 1024 rows, looked back 256 tiles at a time)
against the unfiltered rows: row counts at the edges of a tile, of a window of tiles and of two,
with and without attributes, and point_to_voxel through the remap."""
import numpy as np
import pytest
import torch

from paper_2102_11084_gb300 import vg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 1023, 1024, 1025, 256 * 1024, 256 * 1024 + 1, 600_001])
@pytest.mark.parametrize("channels", [0, 3])
def test_rows_kept(rows, channels):
    # `rows` cells of one to three points each, in any order
    r = np.random.Generator(np.random.PCG64(rows))
    n = r.integers(1, 4, rows)
    cell = np.repeat(np.arange(rows), n)
    cell = cell[r.permutation(len(cell))]
    idx = np.stack([cell % 1000, cell // 1000 % 1000, cell // 1_000_000], 1)
    x = torch.from_numpy(((idx + 0.5) * 0.125).astype(np.float32)).cuda()
    kw = {}
    if channels:
        kw["attrs"] = torch.from_numpy(r.integers(0, 256, (len(cell), 3), np.uint8)).cuda()
    args = ((x, [0, len(cell)]), [0.125])
    a = vg.downsample_frames(*args, point_to_voxel=True, **kw)
    b = vg.downsample_frames(*args, point_to_voxel=True, min_count=2, **kw)
    assert a.keys.numel() == rows
    keep = a.counts.to(torch.int64) >= 2
    assert torch.equal(b.keys, a.keys[keep]) and torch.equal(b.counts, a.counts[keep])
    assert torch.equal(b.centroids, a.centroids[keep])
    assert b.offsets[-1] == int(keep.sum())
    if channels:
        assert torch.equal(b.attrs, a.attrs[keep])
    place = torch.where(keep, torch.cumsum(keep, 0) - 1, torch.full_like(keep, -1, dtype=torch.int64))
    assert torch.equal(b.point_to_voxel.to(torch.int64), place[a.point_to_voxel.to(torch.int64)])
