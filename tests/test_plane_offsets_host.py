"""The 3-D tile kernel addresses a plane by 32-bit byte offsets; the cell such
an offset belongs to (the index of its word) has to be exact up to the largest
plane whose grid fits the device, 2^30 FP32 or 2^29 FP64 cells.  On the CPU:
such a grid takes 160 GB and more."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_cell_of_an_offset_is_exact_on_the_largest_planes(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "plane_offsets"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_2304_05657_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "host", "plane_offsets.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["0", "0"]
