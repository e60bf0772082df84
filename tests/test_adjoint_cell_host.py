"""The hand-derived local adjoints of the direct adjoint step, on the CPU:
the collision's and the WENO3 derivative's against fourth-order central
differences of their forward forms, and the WENO3 partials at the smallest
epsilon (1e-75), where scaling line and epsilon by powers of two must not
change a bit (no intermediate leaves the FP64 range).

Collision: steps of 1e-4 on polynomials with coefficients of order 1 in
arguments of order 0.1 to 1 leave a truncation below 1e-14 and rounding of about
1e-15 / 1e-4: 1e-10 of the largest adjoint.  WENO3: steps of 1e-3 on functions
whose fifth derivatives reach about 1e3 (epsilon 1): 1e-12 * 1e3 / 30, bar
1e-9."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_local_adjoints(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "adjoint_cell"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                    "-Xcompiler", "-ffp-contract=off", "-I", os.path.join(ROOT, "paper_2304_05657_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "adjoint_cell.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    collision, weno, scaled = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert float(collision) <= 1e-10
    assert float(weno) <= 1e-9
    assert int(scaled) == 0
