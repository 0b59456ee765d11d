"""Test-only glue: a harness program linked with the library's own objects and
the stand-in for the CUDA runtime (harness/fake_cuda.cpp) instead of the real one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build(folder, source):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    from paper_2410_23802_gb300 import build as b
    b.build()
    objects = [os.path.join(b.BUILD, f"vlb_{part}.o") for part in ("capi", "lattice", "batch", "particles")]
    for src in (source, "fake_cuda.cpp"):
        objects.append(str(folder / (src + ".o")))
        subprocess.run([nvcc, "-std=c++17", "-O1", "-c", os.path.join(ROOT, "tests", "harness", src), "-o",
                        objects[-1]], check=True)
    exe = str(folder / "harness")
    subprocess.run(["g++", *objects, "-lpthread", "-o", exe], check=True)
    return exe
