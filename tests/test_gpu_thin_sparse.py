"""Thinning of clouds whose points have fewer candidates than the threshold on average: the host
looks whether any is marked before the loop is prepared.  None, a few (one pass, several), and
no valid point, against the oracle; and batches of much of the cloud."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_11084_gb300 import vg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("crowd", [0, 2, 21, 22, 60])
@pytest.mark.parametrize("t,batch", [(20, 3), (20, 1000), (1, 1)])
def test_few_marked(crowd, t, batch):
    rng = np.random.Generator(np.random.PCG64(crowd + batch))
    x = rng.uniform(0, 4.0, (8000, 3)).astype(np.float32)
    if crowd:
        x[100:100 + crowd] = (2.0 + rng.uniform(0, 0.02, (crowd, 3))).astype(np.float32)
    x[::31] = np.nan
    pr = rng.permutation(8000).astype(np.uint32)
    keep, passes, st = oracle.thin(x, 0.05, t, pr, batch=batch)
    assert st == 0
    res = vg.thin(torch.from_numpy(x).cuda(), 0.05, t, torch.from_numpy(pr.view(np.int32)).cuda(),
                  batch=batch)
    assert np.array_equal(res.keep.cpu().numpy(), keep)
    assert res.num_kept == int(keep.sum()) and res.passes == passes


def test_no_valid_point():
    x = torch.full((500, 3), float("nan"), device="cuda")
    res = vg.thin(x, 0.05, 3, torch.arange(500, dtype=torch.int32, device="cuda"))
    assert res.num_kept == 0 and not bool(res.keep.any()) and res.passes == 1


@pytest.mark.parametrize("share", [1, 2, 3, 8])
@pytest.mark.parametrize("n,ext,t", [(20_000, 0.5, 2), (20_000, 0.5, 20), (30_000, 1.2, 2)])
def test_batches_of_much_of_the_cloud(n, ext, t, share):
    # few passes: either side of the line between counts kept and counts taken afresh
    rng = np.random.Generator(np.random.PCG64(n + t))
    x = rng.uniform(0, ext, (n, 3)).astype(np.float32)
    pr = rng.permutation(n).astype(np.uint32)
    keep, passes, st = oracle.thin(x, 0.05, t, pr, batch=n // share)
    assert st == 0
    res = vg.thin(torch.from_numpy(x).cuda(), 0.05, t, torch.from_numpy(pr.view(np.int32)).cuda(),
                  batch=n // share)
    assert np.array_equal(res.keep.cpu().numpy(), keep)
    assert res.num_kept == int(keep.sum()) and res.passes == passes
