"""The kernel that the benchmark names from a handle's step description."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402


@pytest.mark.parametrize("forced,cells,threads,want", [
    (0, 64, 1, "step_tile_kernel"), (0, 32, 1, "step_tile_kernel"), (0, 32, 3, "step_small_kernel"),
    (0, 64, 3, "block_steps_kernel"), (0, 320, 3, "block_steps_kernel"),
    (1, 32, 3, "step_kernel"), (9, 64, 1, "step_kernel_cell")])
def test_step_kernel_name(forced, cells, threads, want):
    info = type("I", (), dict(tile_cells=cells, threads_per_cell=threads))()
    assert bench.step_kernel_name(forced, info) == want
