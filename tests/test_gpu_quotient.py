"""The lattice kernel's reciprocal and quotient on the GPU against extended
precision: Newton's step leaves the square of the approximate reciprocal's
error (2^-46 relative in FP32) and one rounding, the quotient's correction the
same, so both lie within 0.51 units in the last place."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reciprocal_and_quotient_are_within_half_a_unit(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "quotient_gpu")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2410_23802_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "harness", "quotient_gpu.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert out[0] == "fp32" and out[3] == "fp64"
    assert max(float(v) for v in (out[1], out[2])) <= 0.51, out
    assert max(float(v) for v in (out[4], out[5])) <= 0.51, out
