"""Thinning with a radius whose square is not finite in binary32 (every point of a cell is then
a neighbour of every other) or rounds to zero, against the oracle: keep flags, number kept and
passes, with odd and even batches through every form of the loop."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_11084_gb300 import vg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,t,batch", [(700, 300, 7), (700, 300, 8), (701, 300, 33), (64, 3, 1),
                                       (3000, 5, 2999)])
@pytest.mark.parametrize("radius,cell", [(1.0e20, 1.0e20), (3.0e38, 3.0e38), (1.0e-30, 1.0)])
def test_square_beyond_binary32(n, t, batch, radius, cell):
    rng = np.random.Generator(np.random.PCG64(n + batch))
    x = rng.uniform(0, 0.5, (n, 3)).astype(np.float32)
    x[: n // 2] = x[0]  # (neighbours at distance zero too)
    pr = rng.permutation(n).astype(np.uint32)
    keep, passes, st = oracle.thin(x, cell, t, pr, radius=radius, batch=batch)
    assert st == 0
    res = vg.thin(torch.from_numpy(x).cuda(), cell, t, torch.from_numpy(pr.view(np.int32)).cuda(),
                  radius=radius, batch=batch)
    assert np.array_equal(res.keep.cpu().numpy(), keep)
    assert res.num_kept == int(keep.sum()) and res.passes == passes
