"""The step's fast reciprocals against IEEE 1 / x: the FP32 hardware
reciprocal is documented to 1 ulp; the FP64 one takes a seed of relative
error below 2^-19 through x (1 + e + e^2), e = 1 - b x, which leaves e^3 <
2^-57 and the roundings of the last two operations: within 1 ulp."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fast_reciprocals_are_within_one_ulp(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = tmp_path / "reciprocal"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_2304_05657_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "reciprocal.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert int(out[0]) <= 1 and int(out[1]) <= 1, out
