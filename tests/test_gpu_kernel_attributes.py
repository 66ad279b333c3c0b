"""A kernel's attributes belong to the current device and context: a scene builds
on a device whose kernels have none yet, whatever was set or failed elsewhere.

The second device is imitated: a program linked against the library's objects
passes its cudaFuncSetAttribute calls through a wrapper, which takes the shared
memory limit away again between two builds (as a new device has it), or fails
one call.  A launch above the limit is refused by the runtime, on the host."""

import glob
import os
import shutil
import subprocess

import pytest

from paper_2503_23410_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "vafr.h"

#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <vector>

extern "C" cudaError_t __real_cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v);
static const void* limited[16];
static int n_limited = 0, failing = 0;

extern "C" cudaError_t __wrap_cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        if (failing > 0 && failing--) return cudaErrorMemoryAllocation;
        if (n_limited < 16) limited[n_limited++] = f;
    }
    return __real_cudaFuncSetAttribute(f, a, v);
}

static int build(int n) {
    std::vector<float> tris(9 * n);
    for (int k = 0; k < 9 * n; ++k) tris[k] = (float)((k * 7919 + 13) % 1009) / 504.5f - 1.0f;
    const float light[3] = {0.0f, -1.0f, 0.0f};
    vafr_scene* scene = nullptr;
    const int rc = vafr_build_scene(tris.data(), nullptr, n, light, nullptr, &scene);
    if (rc == 0) vafr_scene_destroy(scene);
    return rc;
}

int main(int argc, char** argv) {
    if (argc > 1 && !std::strcmp(argv[1], "fails once")) {
        failing = 1;
        const int first = build(5000), second = build(5000);
        std::printf("%d %d", first != 0, second);
        return 0;
    }
    const int first = build(5000);
    for (int k = 0; k < n_limited; ++k)
        if (__real_cudaFuncSetAttribute(limited[k], cudaFuncAttributeMaxDynamicSharedMemorySize, 0)) return 1;
    const int second = build(5000);
    std::printf("%d %d", first, second);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(V, tmp_path_factory):
    d = tmp_path_factory.mktemp("attributes")
    src, exe = d / "attributes.cu", d / "attributes"
    src.write_text(PROGRAM)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", os.path.join(build.HERE, "..", "include"), "-o", str(exe),
                    str(src), *glob.glob(os.path.join(build.OBJ, "*.o")), "-Xlinker", "--wrap=cudaFuncSetAttribute",
                    "-lpthread", "-ldl", "-lrt"], check=True)
    return str(exe)


@pytest.mark.parametrize("how, want", [("new device", "0 0"), ("fails once", "1 0")])
def test_scenes_build_where_the_attribute_is_not_set_yet(program, how, want):
    r = subprocess.run([program, how], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == want, r.stdout + r.stderr
