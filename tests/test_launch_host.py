"""Which kernels may come in while the one before them runs (programmatic
dependent launch): the lattice kernels read the populations as data nobody
writes while they exist, so two of them may not follow each other that way.  The
library's objects run over a stand-in for the CUDA runtime that records the
launches (harness/launch_host.cpp)."""
import subprocess

import pytest

import host_harness


@pytest.fixture(scope="module")
def launches(tmp_path_factory):
    exe = host_harness.build(tmp_path_factory.mktemp("launch"), "launch_host.cpp")
    runs = {}
    for line in subprocess.run([exe], capture_output=True, text=True, check=True, timeout=120).stdout.splitlines():
        run, kernel, early = line.split()
        runs.setdefault(run, []).append(("lattice" if "lattice" in kernel else "particle", early == "1"))
    return runs


@pytest.mark.parametrize("run", ["alone", "batch"])
def test_lattice_kernels_without_particles_wait(launches, run):
    assert launches[run + "0"] == [("lattice", False)] * 6


@pytest.mark.parametrize("run", ["alone", "batch"])
def test_kernels_behind_particle_kernels_come_in_early(launches, run):
    """A particle kernel lies between any two lattice kernels of one handle."""
    assert all(early for _, early in launches[run + "1"])
    per_step = {"alone": ["particle", "lattice"], "batch": ["particle", "lattice", "lattice"]}[run]
    assert [kind for kind, _ in launches[run + "1"]] == per_step * {"alone": 6, "batch": 3}[run]


@pytest.mark.parametrize("run", ["alone", "batch"])
def test_lattice_kernels_of_crowded_lattices_wait(launches, run):
    """400 disks on 124 tiles: the waiting CTAs would crowd on the SMs that the
    particle kernel leaves free."""
    assert len(launches[run + "2"]) == len(launches[run + "1"])
    assert all(early == (kind == "particle") for kind, early in launches[run + "2"])
