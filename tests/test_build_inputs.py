"""Which device inputs a scene build reads where they lie (csrc/inputs.h, compiled
here): only what is on the build's device, in whole floats, and wholly inside one
allocation.  Everything else is copied, as memory of another device has to be."""

import ctypes
import os
import subprocess

import pytest

from paper_2503_23410_gb300 import build

BASE, SIZE = 0x7f0000000000, 4096


@pytest.fixture(scope="module")
def readable(tmp_path_factory):
    d = tmp_path_factory.mktemp("inputs")
    (d / "inputs.cpp").write_text("""
#include "inputs.h"
extern "C" int readable(int here, unsigned long long at, unsigned long long bytes, unsigned long long base,
                        unsigned long long size) {
    return vafr::readable_in_place(here != 0, at, bytes, base, size);
}
""")
    so = d / "inputs.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(so), str(d / "inputs.cpp")],
                   check=True)
    f = ctypes.CDLL(str(so)).readable
    f.argtypes = [ctypes.c_int] + [ctypes.c_ulonglong] * 4
    return f


@pytest.mark.parametrize("here, at, count, want", [
    (1, BASE, SIZE, 1),
    (1, BASE + 4, SIZE - 4, 1),
    (1, BASE + SIZE, 0, 1),
    (0, BASE, SIZE, 0),              # another device's
    (1, BASE + 2, 36, 0),            # between two floats
    (1, BASE, SIZE + 4, 0),          # longer than the allocation
    (1, BASE + 4, SIZE, 0),
    (1, BASE - 4, 36, 0),
    (1, BASE + SIZE + 4, 0, 0),
    (1, BASE + 4, 2 ** 64 - 4, 0),   # no wrap of the sum
])
def test_in_place(readable, here, at, count, want):
    assert readable(here, at, count, BASE, SIZE) == want


def test_unknown_allocation(readable):
    assert readable(1, BASE, 36, 0, 0) == 0
