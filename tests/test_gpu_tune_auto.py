"""The tuner keeps AUTO where it beats the groupings it reports: a tuned plan is not slower than
one left alone.  Eight camera frames, which the occupancy trie groups in a fraction of the others'
time."""
import numpy as np
import torch
import pytest

from paper_2102_11084_gb300 import synth, vg

pytestmark = pytest.mark.gpu


def test_batch_that_auto_wins(tmp_path):
    frames = [synth.rgbd_frame(640, 480, seed=s) for s in range(4)] * 2
    x = torch.from_numpy(np.concatenate(frames)).cuda()
    n, F = x.shape[0], len(frames)
    offs = [307_200 * f for f in range(F + 1)]
    ref = vg.downsample_frames((x, offs), [0.05] * F)
    d = "cuda"
    b = dict(xyz=x, frame_offsets=torch.tensor(offs, dtype=torch.int64, device=d), n_frames=F,
             origins=torch.zeros((F, 3), device=d), leaves=torch.full((F,), 0.05, device=d),
             out_keys=torch.empty(n, dtype=torch.int64, device=d),
             out_centroids=torch.empty((n, 3), device=d),
             out_counts=torch.empty(n, dtype=torch.int32, device=d),
             out_frame_offsets=torch.zeros(F + 1, dtype=torch.int64, device=d),
             out_error=torch.zeros(1, dtype=torch.int32, device=d))
    s = torch.cuda.Stream()
    plan = vg.Plan(F, n)
    with torch.cuda.stream(s):
        times = plan.tune(**b, reps=3, stream=s)
        assert len(times) == 12 and plan.get()["method"] == "auto"
        plan.run(**b, stream=s)
        s.synchronize()
    assert int(b["out_error"].item()) == 0
    assert b["out_frame_offsets"].cpu().tolist() == ref.offsets
    assert torch.equal(b["out_keys"][:ref.offsets[-1]], ref.keys)
    path = str(tmp_path / "tuned.json")
    plan.save_tuning(path)
    other = vg.Plan(F, n, method="hash")
    other.load_tuning(path)
    assert other.get()["method"] == "auto"
    plan.close()
    other.close()
