"""Forward-mode division (a / b)' = (a' - (a / b) b') / b in FP32 where the two
terms nearly cancel.  With u the unit roundoff, 1 / b and a (1 / b) carry one
rounding each and the product with b' one more: 3 u of the terms; what follows
the cancellation is relative to the small difference (1e-4 of the terms here:
3e-4 u more)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_derivative_of_a_quotient(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "dual_division"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_2304_05657_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "dual_division.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    assert float(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout) <= 3.001
