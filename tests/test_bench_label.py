"""The kernel that the benchmark names from a handle's step description, and the
hash that its committed traffic figures are valid for."""
import os
import shutil
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


def test_the_source_hash_covers_every_step_kernel(tmp_path, monkeypatch):
    csrc = os.path.join(bench.ROOT, "paper_1809_01600_gb300", "csrc")
    copy = tmp_path / "paper_1809_01600_gb300" / "csrc"
    shutil.copytree(csrc, copy)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    shas = {bench.kernel_source_sha()}
    steps = ["lbms_kernels.cuh", "lbms_step_tile.cuh", "lbms_step_small.cuh", "lbms_launch_tile.cu",
             "lbms_launch_small.cu", "lbms_launch.cu", "lbms_step_launch.cuh", "lbms_lattice.cuh", "lbms_internal.h"]
    for f in steps:
        (copy / f).write_text((copy / f).read_text() + "// changed\n")
        shas.add(bench.kernel_source_sha())
    assert len(shas) == 1 + len(steps)
