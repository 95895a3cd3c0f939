"""The chained scans over tiles of 1024 rows, looked back by a warp 32 tiles at a time (the
minimum-count filter) or by the whole block (the pyramid's merges): sizes at the edges of the
warp's window."""
import pytest

from tests import test_gpu_filter_tiles as filter_tiles
from tests import test_gpu_pyramid_tiles as pyramid_tiles

pytestmark = pytest.mark.gpu

ROWS = [31 * 1024 + 1, 32 * 1024, 32 * 1024 + 1, 33 * 1024, 64 * 1024 + 1]


@pytest.mark.parametrize("rows", ROWS)
def test_filter(rows):
    filter_tiles.test_rows_kept(rows, 0)


@pytest.mark.parametrize("rows", ROWS)
def test_pyramid(rows):
    pyramid_tiles.test_tile_edges(rows, 1.0)
