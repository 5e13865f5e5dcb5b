"""The plans of the network's convolutions (conv_plan in kernels_unet.cu) for grids
of 1 to 1024 voxels per axis and every channel count a network can have: boxes
that a TMA copy takes, tiles that cover the grid, shared memory and TMEM that a
CTA has, and tiles put together only where enough groups are left for the SMs.
Host code only: compiled with nvcc, run on the CPU."""
import os
import shutil
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_plans_of_every_grid():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "conv_plan_check")
        subprocess.run([nvcc, "-O1", "-Xptxas", "-O0", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I" + os.path.join(ROOT, "include"), "-o", exe, os.path.join(HERE, "host", "conv_plan_check.cu")],
                       check=True, capture_output=True, text=True)
        out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
