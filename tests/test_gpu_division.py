"""The lattice kernel's reciprocal and quotient are correctly rounded: equal to
the language's division, bit by bit, for operands and results in the normal
range (harness/division_gpu.cu)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reciprocal_and_quotient_are_correctly_rounded(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "division_gpu")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2410_23802_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "harness", "division_gpu.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True, timeout=120).stdout
    assert int(out) == 0
