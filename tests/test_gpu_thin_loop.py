"""The two forms of the thinning loop (counts kept through all passes in one launch, or counted
afresh every pass) against the oracle: keep flags, number kept and passes are whole numbers
and must be equal.  The sizes lie at the edges of the batch search (2048 list entries a step,
one list entry more or less than a batch) and on both sides of the rule that picks the form
(all candidate pairs against the passes a fresh count would take)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2102_11084_gb300 import vg

pytestmark = pytest.mark.gpu


def check(x, cell, t, pr, batch, radius=None):
    keep, passes, st = oracle.thin(x, cell, t, pr, radius=radius, batch=batch)
    assert st == 0
    res = vg.thin(torch.from_numpy(x).cuda(), cell, t, torch.from_numpy(pr.view(np.int32)).cuda(),
                  radius=radius, batch=batch)
    assert np.array_equal(res.keep.cpu().numpy(), keep)
    assert res.num_kept == int(keep.sum()) and res.passes == passes


@pytest.mark.parametrize("n,batch", [(2047, 1), (2048, 2047), (2049, 2048), (4097, 100),
                                     (6000, 1000), (6000, 5999), (6000, 6000)])
@pytest.mark.parametrize("t", [0, 5])
def test_batches_and_list_steps(n, batch, t):
    rng = np.random.Generator(np.random.PCG64(n + batch))
    x = rng.uniform(0, 0.5 if batch > 1 else 0.9, (n, 3)).astype(np.float32)
    x[::97] = np.nan
    check(x, 0.05, t, rng.permutation(n).astype(np.uint32), batch)


@pytest.mark.parametrize("n,t,batch", [(3000, 5, 1500), (3000, 400, 700), (2000, 0, 1999),
                                       (3000, 5, 4), (900, 20, 20)])
def test_dense_clouds_both_sides_of_the_rule(n, t, batch):
    rng = np.random.Generator(np.random.PCG64(n + t))
    x = (1.0 + rng.uniform(0, 0.11, (n, 3))).astype(np.float32)
    check(x, 0.05, t, rng.permutation(n).astype(np.uint32), batch, radius=0.04)


def test_recounted_form():
    # 24,000 points of a few cells, two passes: a fresh count stops at the third neighbour
    rng = np.random.Generator(np.random.PCG64(11))
    x = (1.0 + rng.uniform(0, 0.04, (24_000, 3))).astype(np.float32)
    check(x, 0.05, 2, rng.permutation(24_000).astype(np.uint32), 23_000)


def test_equal_and_large_priorities():
    rng = np.random.Generator(np.random.PCG64(7))
    x = rng.uniform(0, 0.3, (3000, 3)).astype(np.float32)
    check(x, 0.05, 3, np.zeros(3000, np.uint32), 50)
    check(x, 0.05, 3, rng.integers(0xfffffff0, 1 << 32, 3000, dtype=np.uint64).astype(np.uint32),
          50)


@pytest.mark.parametrize("n,ext,t,batch", [
    (20_000, 0.4, 10, 4096), (20_000, 0.4, 10, 4097),  # either side of a block's own lists
    (1_500, 0.14, 3, 1), (6_000, 0.2, 0, 33),          # most list entries unmarked at the end
    (60_000, 1.0, 20, 4000),                           # groups of several rounds, lists shared
    (40_000, 1.6, 1, 500),                             # few candidates: scattered
])
def test_forms_of_the_kept_counts(n, ext, t, batch):
    rng = np.random.Generator(np.random.PCG64(n + batch))
    x = rng.uniform(0, ext, (n, 3)).astype(np.float32)
    x[: n // 8] *= 0.3  # crowded cells among sparse ones
    x[::211] = np.inf
    check(x, 0.05, t, rng.permutation(n).astype(np.uint32), batch)
