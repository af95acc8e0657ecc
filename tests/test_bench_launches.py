"""The bench's count of an FP32 render's launches (CPU only), on rounds counted by hand."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


@pytest.mark.parametrize("live,n_rays,n_cells,tail,want", [
    ([900], 1000, 512, 1000, 1 + 3 + 4),  # one round of the tail: scan, scatter, tail
    ([900], 1000, 512, -1, 1 + 4 + 4),  # one round of tiles, whose rays all ended: with the (idle) tail
    ([900, 300, 0], 1000, 4096, -1, 1 + 3 * 4 + 2 + 4),
    ([900, 300], 1000, 4096, 500, 1 + 2 * 4 + 1 + 4),  # the second round ended by its own tail
    ([900, 300, 20], 1000, 4096, 500, 1 + 2 * 4 + 3 + 2 + 4),  # ... but for rays waiting in empty voxels: a third
    ([900, 300, 0], 1000, 4097, -1, 1 + 3 * 5 + 2 + 4),  # the scan in two launches
    ([50] * 87, 1 << 24, 32768, 20, 1 + 87 * 5 + 86 + 4),
])
def test_launches_by_hand(live, n_rays, n_cells, tail, want):
    import bench
    assert bench.fp32_launches(live, n_rays, n_cells, tail) == want
