"""The benchmark reports measured DRAM traffic only for the tiles and the grid size that
were captured (CPU)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("tile,key", [([64, 8, 19], "stream3d_pair"), ([32, 16, 19], None)])
def test_the_record_belongs_to_the_captured_tile(tile, key):
    assert bench.step_kernel_name(dict(step_kernel=2, tile=tile), 3) == ("stream3d_pair_kernel", key)


@pytest.mark.parametrize("key", sorted(bench.NCU_TRAFFIC))
def test_the_record_belongs_to_the_captured_size(key):
    rec = bench.NCU_TRAFFIC[key]
    assert bench.ncu_traffic(key, rec["nodes"]) == rec["bytes"]
    for nodes in (106 * 200 * 200, rec["nodes"] - 1, 2 * rec["nodes"]):
        assert bench.ncu_traffic(key, nodes) is None
