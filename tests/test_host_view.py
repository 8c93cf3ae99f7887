"""Which host arrays the kernels of lce_bconv2d_host access themselves and which they leave to the copy engine: the rule
of csrc/host_view.cuh, compiled for the host and called with what the driver would say of an address."""
import ctypes
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2011_09398_b200" / "csrc"

SHIM = """
#include "host_view.cuh"
extern "C" uint64_t view(uint64_t array, int pinned, uint64_t device) { return lce::kernel_view(array, lce::HostMemory{pinned != 0, device}); }
"""


@pytest.fixture(scope="module")
def view(tmp_path_factory):
    where = tmp_path_factory.mktemp("host_view")
    (where / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(where / "shim.so"), str(where / "shim.cpp")], check=True)
    fn = ctypes.CDLL(str(where / "shim.so")).view
    fn.restype = ctypes.c_uint64
    fn.argtypes = [ctypes.c_uint64, ctypes.c_int, ctypes.c_uint64]
    return fn


BASE = 0x7F5100000000


def test_pinned_arrays_on_whole_words_are_the_kernels(view):
    for offset in (0, 4, 8, 12, 16, 4096 + 4):
        assert view(BASE + offset, 1, BASE + offset) == BASE + offset
    assert view(BASE, 1, 0x1000) == 0x1000      # the device's address is the one that counts where the two differ


def test_pageable_arrays_are_the_copy_engines(view):
    assert view(BASE, 0, 0) == 0
    assert view(BASE, 0, BASE) == 0


@pytest.mark.parametrize("offset", [1, 2, 3, 5, 17, 18])
def test_arrays_that_do_not_start_on_a_word_are_the_copy_engines(view, offset):
    assert view(BASE + offset, 1, BASE + offset) == 0
    assert view(BASE + offset, 1, BASE) == 0 and view(BASE, 1, BASE + offset) == 0
