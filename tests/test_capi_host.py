"""The C ABI's host code compiled against a stand-in for the CUDA runtime that
keeps no more order between copies and streams than CUDA promises
(harness/fake_cuda.cpp, capi_host.cu): what it allocates and in which order it copies."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    folder = tmp_path_factory.mktemp("capi")
    csrc = os.path.join(ROOT, "paper_2410_23802_gb300", "csrc")
    harness = os.path.join(ROOT, "tests", "harness")
    objects = []
    for src in (os.path.join(csrc, "vlb_capi.cu"), os.path.join(harness, "capi_host.cu"),
                os.path.join(harness, "fake_cuda.cpp")):
        objects.append(str(folder / (os.path.basename(src) + ".o")))
        subprocess.run([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-gencode",
                        "arch=compute_103a,code=sm_103a", "-I", csrc, "-c", src, "-o", objects[-1]], check=True)
    exe = str(folder / "capi_host")
    subprocess.run(["g++", *objects, "-lpthread", "-o", exe], check=True)
    return exe


def _check(harness, name):
    r = subprocess.run([harness, name], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr


def test_loaded_image_is_saved_again(harness):
    _check(harness, "roundtrip")
