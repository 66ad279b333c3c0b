"""Kernels launched with overlap begin while the launch before them still writes.
What that one writes -- LP texels, lumas, depths, hole and tile lists, the
triangle-to-leaf table -- may not be read through the read-only path (__ldg,
ld.global.nc, const __restrict__), which CUDA allows only for memory that is
constant for the kernel's whole life."""

import os
import re

import pytest

from paper_2503_23410_gb300 import build

# what a kernel of the file's overlapped launches reads of earlier launches' output
WRITTEN = {
    "fxaa.cu": r"\blp\b|\blum\b|\bluma\b|\blp_aa\b",
    "reconstruct.cu": r"\blp\b|\blp_aa\b",
    "reproject.cu": r"\blp\b|\bdepth\b|\bvert\b|\bzbuf\b|\bholes\b",
    "raster.cu": r"\bbig\b|\bbig_leaf\b|\bbig_first\b|\bleaf_of\b|\bvbuf\b|\bcounter\b",
    "render.cu": r"\bcount\b",
    "tree4.cu": r"\bstate\b|\bcounts\b|\bfates\b|\bclusters[01]?\b|\bscanned\b",
}


def _text(name):
    src = open(os.path.join(build.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", src)


def _calls(src, name):
    """The argument text of every call of `name`."""
    for m in re.finditer(name + r"\(", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        yield src[m.end():i - 1]


def _body(src, kernel):
    i = src.index("{", re.search(r"\b" + kernel + r"\([^;{]*\{", src).start())
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        j += 1
    return src[i:j]


@pytest.mark.parametrize("name", sorted(WRITTEN))
def test_no_read_only_loads_of_written_memory(name):
    src = _text(name)
    assert "after_previous()" in src
    bad = [c for c in _calls(src, "__ldg") if re.search(WRITTEN[name], c)]
    assert not bad, bad
    # inline read-only loads are of tables: their address is a parameter that is never an LP buffer
    for m in re.finditer(r'asm[^;]*ld\.global\.nc[^;]*;', src):
        assert not re.search(WRITTEN[name], m.group(0)), m.group(0)


def test_no_restricted_parameters_of_overlapped_kernels():
    for name in WRITTEN:
        src = _text(name)
        for m in re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\(([^{;]*)\)\s*\{", src):
            if "after_previous()" in _body(src, m.group(1)):
                assert "__restrict__" not in m.group(2), (name, m.group(1))


def test_the_hole_list_is_read_plainly():
    """The hole cast's work items come from the launch before it, not from the layout."""
    assert not re.search(r"lp_ray\(f, \(int\)w,", _body(_text("render.cu"), "k_render_list"))
    assert re.search(r"lp_ray\(f, f\.work\[", _body(_text("render.cu"), "k_render_list"))
    assert "__ldg(f.work" not in _body(_text("render.cu"), "k_render_list")
