"""The lattice kernel's wall rules (compiled for the host) against the rules as
the paper's readings state them, direction by direction: every combination of
periodic, closed and open sides, lattices of 2, 3 and 5 cells a side, every
cell and direction."""
import itertools
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)


def _rule(nx, ny, per, opened, x, y, i):
    """(bounces, off a y side, source x, source y): the source x - e_i wraps on a
    periodic axis and moves back across an open side; across a closed side the
    population bounces back, corners between closed sides off the y side."""
    sx, sy = x - EX[i], y - EY[i]
    out_x = out_y = False
    if per[0]:
        sx %= nx
    else:
        out_x = not 0 <= sx < nx
    if per[1]:
        sy %= ny
    else:
        out_y = not 0 <= sy < ny
    if out_x and opened[0 if sx < 0 else 1]:
        sx, out_x = x, False
    if out_y and opened[2 if sy < 0 else 3]:
        sy, out_y = y, False
    return (out_x or out_y, out_y, *((x, y) if out_x or out_y else (sx, sy)))


def test_host_compiled_wall_rules(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "pull_host")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-x", "cu", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2410_23802_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "harness", "pull_host.cu"), "-o", exe], check=True)
    axis = [(1, 0, 0)] + [(0, a, b) for a in (0, 1) for b in (0, 1)]  # periodic, or each end closed / open
    rows, want = [], []
    for nx, ny, ax, ay in itertools.product((2, 3, 5), (2, 3, 5), axis, axis):
        opened = (ax[1], ax[2], ay[1], ay[2])
        for y, x, i in itertools.product(range(ny), range(nx), range(9)):
            rows.append((nx, ny, ax[0], ay[0], *opened, x, y, i))
            bounce, off_y, sx, sy = _rule(nx, ny, (ax[0], ay[0]), opened, x, y, i)
            want.append((int(bounce), int(off_y), sy * (nx + 3) + sx))
    out = subprocess.run([exe], input="\n".join(" ".join(map(str, r)) for r in rows) + "\n", capture_output=True,
                         text=True, check=True).stdout.split("\n")
    got = [tuple(map(int, line.split())) for line in out if line]
    assert len(got) == len(want)
    bad = [(r, g, w) for r, g, w in zip(rows, got, want) if g != w]
    assert not bad, bad[:5]
