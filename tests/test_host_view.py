"""Which host arrays the kernels of lce_bconv2d_host access themselves and which they leave to the copy engine: the rule
of csrc/host_view.cuh, compiled for the host and called with what the driver would say of an address."""
import ctypes
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2011_09398_b200" / "csrc"

SHIM = """
#include "host_view.cuh"
extern "C" uint64_t view(uint64_t array, uint64_t bytes, int write, int pinned, uint64_t device, uint64_t first, uint64_t range, int writable)
{
    return lce::kernel_view(array, bytes, write != 0, lce::HostMemory{pinned != 0, device, first, range, writable != 0});
}
"""
BASE, RANGE = 0x7F5100000000, 1 << 20   # a pinned range


@pytest.fixture(scope="module")
def view(tmp_path_factory):
    where = tmp_path_factory.mktemp("host_view")
    (where / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(where / "shim.so"), str(where / "shim.cpp")], check=True)
    fn = ctypes.CDLL(str(where / "shim.so")).view
    fn.restype = ctypes.c_uint64
    fn.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int, ctypes.c_int, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int]

    def call(array, nbytes, write=0, pinned=1, device=None, first=BASE, size=RANGE, writable=1):
        return fn(array, nbytes, write, pinned, array if device is None else device, first, size, writable)
    return call


def test_pinned_arrays_on_whole_words_are_the_kernels(view):
    for offset in (0, 4, 8, 12, 16, 4096 + 4):
        for write in (0, 1):
            assert view(BASE + offset, 4096, write) == BASE + offset
    # the device's address is the one that counts where the two differ
    assert view(0x10000, RANGE, device=BASE) == BASE
    assert view(0x10000, RANGE - 4, device=BASE + 4) == BASE + 4


def test_pageable_arrays_are_the_copy_engines(view):
    assert view(BASE, 4096, pinned=0) == 0
    assert view(BASE, 4096, pinned=0, device=0, first=0, size=0) == 0
    assert view(BASE, 4096, device=0) == 0      # pinned, but not mapped


@pytest.mark.parametrize("offset", [1, 2, 3, 5, 17, 18])
def test_arrays_that_do_not_start_on_a_word_are_the_copy_engines(view, offset):
    assert view(BASE + offset, 4096) == 0
    assert view(BASE + offset, 4096, device=BASE) == 0 and view(BASE, 4096, device=BASE + offset) == 0


def test_arrays_that_leave_their_pinned_range_are_the_copy_engines(view):
    assert view(BASE, RANGE) == BASE and view(BASE, RANGE + 4) == 0                              # only the front is registered
    assert view(BASE + 64, RANGE - 64) == BASE + 64 and view(BASE + 64, RANGE - 60) == 0
    assert view(BASE + RANGE - 4, 4) == BASE + RANGE - 4 and view(BASE + RANGE - 4, 8) == 0
    assert view(BASE + RANGE, 4) == 0 and view(BASE - 4, 8) == 0 and view(BASE + 8 * RANGE, 4) == 0
    assert view(BASE, 2 ** 64 - 4) == 0 and view(BASE + 64, 2 ** 64 - 64) == 0                   # sums that would wrap


def test_memory_the_device_may_only_read_is_not_written_by_a_kernel(view):
    assert view(BASE, 4096, write=0, writable=0) == BASE
    assert view(BASE, 4096, write=1, writable=0) == 0
