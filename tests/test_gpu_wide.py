"""Keys wider than 32 bits under AUTO, in a scan's order and shuffled: the trie or the sort path,
by what sampled neighbours tell; either gives the radix sort's rows bit for bit."""
import numpy as np
import pytest
import torch

from paper_2102_11084_gb300 import vg
from tests._parity import gpu_counts, gpu_keys, to_np

pytestmark = pytest.mark.gpu


def same(a, b):
    assert np.array_equal(gpu_keys(a.keys), gpu_keys(b.keys))
    assert np.array_equal(gpu_counts(a.counts), gpu_counts(b.counts))
    assert np.array_equal(to_np(a.centroids).view(np.int32), to_np(b.centroids).view(np.int32))
    if a.point_to_voxel is not None:
        assert torch.equal(a.point_to_voxel, b.point_to_voxel)


def scan(n, seed, shuffled):
    """Rings on the ground and on a wall of a 150 m site, neighbours some centimetres apart."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.arange(n, device="cuda", dtype=torch.float64)
    a, d = t * 0.0021, 3.0 + 70.0 * (t / n)
    x = torch.stack((75 + d * torch.cos(a), 75 + d * torch.sin(a), 0.002 * d * torch.sin(7 * a)), 1)
    x[::3, 0] = 75.0 + (x[::3, 0] > 75).double() * 60.0
    x = (x + 0.004 * torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)).float()
    x[::17] = float("nan")
    if shuffled:
        x = x[torch.randperm(n, generator=g, device="cuda")]
    return x.contiguous()


def check(x, leaf, **kw):
    for p2v in (False, True):
        same(vg.downsample(x, leaf, point_to_voxel=p2v, **kw),
             vg.downsample(x, leaf, point_to_voxel=p2v, method="sort_lsd", **kw))


@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("leaf", [0.02, 0.004])
@pytest.mark.parametrize("n", [2_621_441, 4_194_304])
def test_above_what_the_trie_always_takes(n, leaf, shuffled):
    check(scan(n, 3, shuffled), leaf)


def uniform(n, seed, cells, leaf):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    i = torch.randint(0, cells, (n, 3), generator=g, device="cuda")
    return ((i + 0.25 * torch.randint(0, 4, (n, 3), generator=g, device="cuda")).float() * leaf)


# prefixes nearly as many as the points from the first level on, or a few points each
@pytest.mark.parametrize("n", [33, 30_001, 1_000_003, 2_621_440])
@pytest.mark.parametrize("bits", [12, 14, 17, 21])
def test_sparse_cells(n, bits):
    leaf = 2.0 ** -bits
    x = uniform(n, bits, 2 ** bits, leaf)  # (dyadic: indices exact)
    x[: n // 8] = x[n // 2: n // 2 + n // 8]     # cells of two and more points, far apart
    x[n // 3] = float("nan")
    check(x.contiguous(), leaf, origin=torch.zeros(3, device="cuda"))


def test_frames_of_sparse_cells():
    leaf = 2.0 ** -16
    x = uniform(900_000, 4, 2 ** 16, leaf)
    offs = [0, 0, 300_001, 300_001, 750_000, 900_000]
    rgb = (torch.arange(3 * x.shape[0], device="cuda") * 37 % 256).to(torch.uint8).reshape(-1, 3)
    for kw in ({}, {"point_to_voxel": True}, {"attrs": rgb, "min_count": 2}):
        a = vg.downsample_frames((x, offs), [leaf] * 5, **kw)
        b = vg.downsample_frames((x, offs), [leaf] * 5, method="sort_lsd", **kw)
        assert a.offsets == b.offsets
        same(a, b)
        assert a.attrs is None or torch.equal(a.attrs, b.attrs)
