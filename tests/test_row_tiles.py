"""The tiles of the kernels that run along rows (row_tiles.h): every cell of a box
once, whatever its row length, and never more than twice the warp rounds of a
walk over the flat cells, so that boxes with short rows don't leave the lanes
idle.  Host code only: compiled with nvcc, run on the CPU."""
import os
import shutil
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_tiles_cover_boxes_of_any_row_length():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "row_tiles_check")
        subprocess.run([nvcc, "-O2", "-std=c++17", "-o", exe, os.path.join(HERE, "host", "row_tiles_check.cu")],
                       check=True, capture_output=True)
        out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
