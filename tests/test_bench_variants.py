"""bench.py's picture of the render variants is the library's: which casts are
longest-first, and which variants have a full-resolution kernel of their own."""

import os
import re

import pytest

import bench
from paper_2503_23410_gb300 import build


def _constant(name):
    src = open(os.path.join(build.CSRC, "vafr_internal.cuh")).read()
    return int(re.search(r"constexpr int %s = (\d+);" % name, src).group(1))


@pytest.mark.parametrize("variant", range(8))
def test_longest_first(variant):
    line = _constant("kPlainTris")
    for n in (1, line, line + 1, 2_000_000):
        want = variant in (_constant("kLptVariant"), _constant("kLptVariantLean")) or (variant == 0 and n > line)
        assert bench.longest_first(variant, n) == want


def test_the_full_resolution_search_times_every_kernel():
    """Variant 0 has one of its own in small scenes; 6 and 7 cast with variant 4's."""
    n = _constant("kNumRenderVariants")
    assert set(bench.gt_variants(n)) == set(range(n)) - {_constant("kLptVariant"), _constant("kLptVariantLean")}
