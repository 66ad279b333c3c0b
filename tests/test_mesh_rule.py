"""The mesh rule of VaFR_Rep as the kernels compile it (csrc/mesh_rule.h, built here
for the host) against the rule in unbounded integers, on both sides of the ring
size from which it takes 64 bits."""

import ctypes
import os
import random
import subprocess

import pytest

from paper_2503_23410_gb300 import build


@pytest.fixture(scope="module")
def ring_partner(tmp_path_factory):
    d = tmp_path_factory.mktemp("mesh_rule")
    (d / "rule.cpp").write_text("""
#include "mesh_rule.h"
extern "C" int partner(int n, int n2, int j, int s) { return vafr::ring_partner(n, n2, j, s); }
""")
    so = d / "rule.so"
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(so),
                    str(d / "rule.cpp")], check=True)
    return ctypes.CDLL(str(so)).partner


def _rule(n, n2, j, s):
    a = (2 * j + 3) * n2
    # largest odd multiple q n of n with q n < a (s = 0) or <= a (s = 1): k = (q - 1) / 2
    q = (a - 1) // n if s == 0 else a // n
    return ((q - 1) // 2) % n2


@pytest.mark.parametrize("s", [0, 1])
def test_same_texel(ring_partner, s):
    rng = random.Random(5)
    rings = [1, 2, 3, 4, 7, 8, 100, 4000, 32766, 32767, 32768, 32769, 65535, 65536, 1 << 20]
    cases = [(n, n2, j) for n in rings for n2 in rings for j in {0, 1, n // 2, n - 2, n - 1} if 0 <= j < n]
    for _ in range(20000):
        n = rng.randint(1, rng.choice([40, 2000, 32770, 100000]))
        n2 = max(1, rng.choice([n, n - rng.randint(0, 40), n + rng.randint(0, 40), rng.randint(1, 100000)]))
        cases.append((n, n2, rng.randrange(n)))
    for n, n2, j in cases:
        assert ring_partner(n, n2, j, s) == _rule(n, n2, j, s), (n, n2, j)


def test_the_kernels_use_it():
    src = open(os.path.join(build.CSRC, "reproject.cu")).read()
    body = src[src.index("bool rep_triangle("):]
    assert "ring_partner(a.y, b.y, j, s)" in body[:body.index("\n}")]
