"""The random bits of stochastic rounding (compiled for the host): the bits that
the nine populations of a cell draw are uncorrelated, so that their rounding
errors do not add up in the cell's mass.  FP16 rounds by the low 13 bits of a
half word, BF16 by all 16.  Over 2^18 keys a correlation of independent bits has
a standard deviation of 0.002; a pair of low halves reaches 0.09."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bits(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("bits") / "random_bits_host")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2410_23802_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "harness", "random_bits_host.cu"), "-o", exe], check=True)
    keys = np.random.default_rng(7).integers(0, 2 ** 32, size=1 << 18, dtype=np.uint64)
    out = subprocess.run([exe], input="\n".join(map(str, keys)) + "\n", capture_output=True, text=True, check=True).stdout
    return np.array(out.split(), dtype=np.uint32).reshape(-1, 9)


@pytest.mark.parametrize("width", [13, 16])
@pytest.mark.parametrize("which", [0, 1])  # f, g
def test_bits_of_a_cell_are_uncorrelated(bits, which, width):
    half = (bits >> (16 * which)) & ((1 << width) - 1)
    c = np.corrcoef(half.T.astype(np.float64)) - np.eye(9)
    assert np.abs(c).max() < 0.03
    assert np.abs(half.mean(axis=0) / (1 << width) - 0.5).max() < 0.003
