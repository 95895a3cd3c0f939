"""Calls whose cooperative launch the device cannot hold (SMs withheld from the process, here by
the library's own limit) take their other routes, with the same results: AUTO the sort path,
the radix passes a launch each, thinning the counts taken afresh every pass."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_11084_gb300 import synth, vg

pytestmark = pytest.mark.gpu


@pytest.fixture
def limit():
    yield vg.lib().vg_debug_set_cooperative_blocks
    vg.lib().vg_debug_set_cooperative_blocks(0)


def same(a, b):
    for x, y in zip(a, b):
        if isinstance(x, torch.Tensor):
            assert torch.equal(x, y)


@pytest.mark.parametrize("n", [20_011, 2_700_001])
@pytest.mark.parametrize("leaf", [0.05, 0.0005])
def test_decimation(limit, n, leaf):
    x = torch.from_numpy(synth.fused_map(n, seed=2, extent=(10.0, 10.0, 3.0))).cuda()
    rgb = (torch.arange(3 * n, device="cuda") * 37 % 256).to(torch.uint8).reshape(-1, 3)
    calls = [lambda m=m, kw=kw: vg.downsample(x, leaf, method=m, **kw)
             for m in ("auto", "sort_lsd", "hash")
             for kw in ({}, {"point_to_voxel": True})]
    calls += [lambda: vg.downsample(x, leaf, attrs=rgb, min_count=2)]
    for call in calls:
        ref = call()
        limit(1)
        got = call()
        limit(0)
        same(got, ref)
    ref = vg.pyramid(x, 0.05, 3)
    limit(1)
    for a, b in zip(vg.pyramid(x, 0.05, 3), ref):
        same(a, b)


def test_voxel_map(limit):
    x = torch.from_numpy(synth.fused_map(50_000, seed=2, extent=(10.0, 10.0, 3.0))).cuda()
    m = vg.VoxelMap(100_000, [-20.0, -20.0, -20.0], 0.05)
    m.insert(x)
    ref = m.extract()
    limit(1)
    same(m.extract(), ref)


@pytest.mark.parametrize("n,ext,t,batch", [(6000, 0.5, 5, 1000), (20_000, 0.4, 10, 4097),
                                           (3000, 0.3, 3, 50), (2000, 0.5, 10 ** 6, 10)])
def test_thinning(limit, n, ext, t, batch):
    # batches of both kept forms, many passes and one
    rng = np.random.Generator(np.random.PCG64(n + batch))
    x = rng.uniform(0, ext, (n, 3)).astype(np.float32)
    x[::97] = np.nan
    pr = rng.permutation(n).astype(np.uint32)
    keep, passes, st = oracle.thin(x, 0.05, t, pr, batch=batch)
    assert st == 0
    limit(1)
    for _ in range(2):
        res = vg.thin(torch.from_numpy(x).cuda(), 0.05, t,
                      torch.from_numpy(pr.view(np.int32)).cuda(), batch=batch)
        assert np.array_equal(res.keep.cpu().numpy(), keep)
        assert res.num_kept == int(keep.sum()) and res.passes == passes
