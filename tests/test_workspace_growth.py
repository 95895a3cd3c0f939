"""A workspace sized for the largest cloud holds what every smaller one's fastest grouping takes:
no workspace query falls as the cloud grows (the serving loop, the cloud pipeline and any C
program size theirs by the largest).  Host functions only."""
import ctypes

import pytest

from paper_2102_11084_gb300 import build as vgbuild
from paper_2102_11084_gb300 import vg

# either side of every size at which AUTO's buffers change, and between
EDGES = [(5 << 19), 1 << 22, 1 << 24]
SIZES = sorted({n for e in EDGES for n in (e - 1, e, e + 1, e + e // 3)} | {0, 1, 1000, 307_200,
               7_700_000, 50_000_000, vg.MAX_POINTS})


@pytest.fixture(scope="module", autouse=True)
def built():
    vgbuild.build()


def grows(query):
    got = [int(query(n)) for n in SIZES]
    assert all(0 < a <= b for a, b in zip(got, got[1:])), list(zip(SIZES, got))


@pytest.mark.parametrize("method", ["auto", "sort", "sort_lsd", "frame", "hash"])
@pytest.mark.parametrize("frames", [1, 16, vg.MAX_FRAMES])
def test_clouds_and_batches(method, frames):
    f = vg.method_flag(method)
    grows(lambda n: vg.lib().vg_downsample_workspace_bytes(n, f))
    grows(lambda n: vg.lib().vg_batch_workspace_bytes(n, frames, f))


@pytest.mark.parametrize("attrs", [None, 256])
@pytest.mark.parametrize("min_count", [1, 2])
def test_extras(attrs, min_count):
    ex = vg.VoxelExtras(attrs, 3 if attrs else 0, attrs, min_count)
    grows(lambda n: vg.lib().vg_downsample_ex_workspace_bytes(n, 4, 0, ctypes.byref(ex)))


@pytest.mark.parametrize("levels", [1, 4])
def test_pyramid(levels):
    grows(lambda n: vg.lib().vg_pyramid_workspace_bytes(n, levels, 0))
