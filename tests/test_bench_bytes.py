"""The bytes that the benchmark bills a run's traversal with."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("nodes,boxes,tris,grid", [(1000, 1000, 700, True), (1000, 1003, 700, True),   # a tie went to the tree
                                                   (1000, 2000, 700, False), (1000, 3600, 700, False)])
def test_grid_runs_are_billed_by_cells_and_tree_runs_by_nodes(nodes, boxes, tris, grid):
    want = bench.CELL_BYTES * nodes + bench.CELL_TRI_BYTES * tris if grid else bench.NODE_BYTES * nodes + bench.TRI_BYTES * tris
    assert bench.structure_bytes(nodes, boxes, tris) == want
