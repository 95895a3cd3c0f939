"""A given origin that is not finite places no point: every valid point's index is out of
range, and every method, entry point and number of frames reports it (as the oracle does)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_11084_gb300 import synth, vg

pytestmark = pytest.mark.gpu

METHODS = ["auto", "sort", "sort_lsd", "hash", "frame"]


@pytest.fixture(scope="module")
def cloud():
    return synth.random_cloud(5000, seed=3, extent=2.0, nan_frac=0.05)


def origin(axis, value):
    o = np.full(3, -1.0, np.float32)
    o[axis] = value
    return o


def refused(call):
    with pytest.raises(vg.VGError) as e:
        call()
    assert e.value.status == vg.Status.RANGE


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_one_cloud(cloud, axis, value):
    o = origin(axis, value)
    assert oracle.downsample(cloud, 0.05, o).status != 0
    x, og = torch.from_numpy(cloud).cuda(), torch.from_numpy(o).cuda()
    for m in METHODS:
        refused(lambda: vg.downsample(x, 0.05, og, method=m))
        refused(lambda: vg.downsample(x, 0.05, og, method=m, point_to_voxel=True))
    refused(lambda: vg.downsample(x, 0.05, og, min_count=2))
    refused(lambda: vg.downsample_noalloc(x, 0.05, og))
    refused(lambda: vg.pyramid(x, 0.05, 3, og))
    prio = torch.arange(len(cloud), dtype=torch.int32, device="cuda")
    refused(lambda: vg.thin(x, 0.05, 5, prio, origin=og))


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("method", METHODS)
def test_one_of_several_frames(cloud, method, value):
    x = torch.from_numpy(cloud).cuda()
    ogs = np.stack([origin(0, -1.0), origin(1, value)])
    refused(lambda: vg.downsample_frames((x, [0, 2000, 5000]), [0.05, 0.1], ogs, method=method))
