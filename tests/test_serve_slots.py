"""Slots of a serving loop with a memory budget: as many as the sort path's workspace allows (the
default grouping's is larger), the larger workspace only where the budget holds it."""
import numpy as np
import pytest
import torch

from paper_2102_11084_gb300 import serve, synth, vg


@pytest.mark.parametrize("budget,want", [
    (None, [500] * 3), (10 ** 6, [500] * 3), (1800, [500] * 3), (1799, [500, 500, 100]),
    (1000, [500, 100, 100]), (999, [100] * 3), (600, [100] * 3), (599, [100, 100]),
    (400, [100, 100]), (399, [100]), (1, [100]), (0, [100]), (1400, [500, 500, 100])])
def test_workspaces(budget, want):
    assert serve.slot_workspaces(3, 100, 500, 100, budget) == want


def test_one_workspace_size():
    assert serve.slot_workspaces(3, 100, 100, 100, 450) == [100, 100]
    assert serve.slot_workspaces(0, 100, 100, 100, None) == [100]


@pytest.mark.gpu
def test_budget_of_three_least_slots():
    frames = [synth.rgbd_frame(160, 120, seed=s) for s in range(6)]
    n, F = 40_000, 4
    least = int(vg.lib().vg_batch_workspace_bytes(n, F, vg.METHOD_SORT))
    budget = 3 * (serve._Slot.other_bytes(n, F) + least)
    srv = serve.Server(max_points=n, max_frames=F, n_slots=3, mem_budget=budget)
    assert len(srv.slots) == 3 and srv.device_bytes == budget
    got = [srv.submit(0, x, 0.05) for x in frames]
    for x, f in zip(frames, got):
        ref = vg.downsample(torch.from_numpy(x).cuda(), 0.05)
        assert np.array_equal(f.result().keys, ref.keys.cpu().numpy().view(np.uint64))
        assert np.array_equal(f.result().centroids, ref.centroids.cpu().numpy())
    srv.close()
    srv = serve.Server(max_points=n, max_frames=F, n_slots=3)
    assert all(s.workspace.numel() > least for s in srv.slots)
    srv.close()
