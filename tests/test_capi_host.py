"""The C ABI's host code over a stand-in for the CUDA runtime that keeps no more
order between copies and streams than CUDA promises (harness/fake_cuda.cpp,
capi_host.cpp): what it allocates and in which order it copies."""
import subprocess

import pytest

import host_harness


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    return host_harness.build(tmp_path_factory.mktemp("capi"), "capi_host.cpp")


def _check(harness, name):
    r = subprocess.run([harness, name], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr


def test_loaded_image_is_saved_again(harness):
    _check(harness, "roundtrip")


def test_device_bytes_counts_every_allocation(harness):
    _check(harness, "footprint")


def test_images_allocate_nothing_on_the_device(harness):
    _check(harness, "full")


def test_fields_are_read_when_helper_threads_get_no_buffer(harness):
    _check(harness, "helpers")
