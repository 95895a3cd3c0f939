"""Attribute means divide exact sums in binary32 below 2^24, where FP64 rounded to float32 gives
the same bits, and in FP64 from there on: sums on either side of the line and counts whose
quotients lie near a rounding boundary, equal to FP64's in numpy bit for bit."""
import numpy as np
import pytest
import torch

from paper_2102_11084_gb300 import vg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("channels", [1, 3, 4])
def test_bits_of_the_quotients(channels):
    # 255 * 65,793 is 2^24 - 1; one point more passes it
    counts = [65_793, 65_794, 65_792, 100_000] + list(range(1, 400))
    r = np.random.Generator(np.random.PCG64(channels))
    cell = np.repeat(np.arange(len(counts)), counts)
    at = r.integers(0, 256, (len(cell), channels), np.uint8)
    at[cell < 3] = 255
    perm = r.permutation(len(cell))
    cell, at = cell[perm], at[perm]
    x = np.stack([(cell + 0.5) * 0.5, np.full(len(cell), 0.25), np.full(len(cell), 0.25)], 1)
    res = vg.downsample(torch.from_numpy(x.astype(np.float32)).cuda(), 0.5,
                        torch.zeros(3, device="cuda"), attrs=torch.from_numpy(at).cuda())
    sums = np.zeros((len(counts), channels), np.int64)
    np.add.at(sums, cell, at.astype(np.int64))
    want = (sums.astype(np.float64) / np.asarray(counts, np.float64)[:, None]).astype(np.float32)
    assert np.array_equal(res.counts.cpu().numpy(), np.asarray(counts))
    assert np.array_equal(res.attrs.cpu().numpy().view(np.int32), want.view(np.int32))
