"""Kernel attributes and occupancy counts are kept per device (csrc/device_once.cuh): the header
compiled against a fake CUDA runtime with several devices, and the library's sources, which must
set attributes nowhere else."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1603_04334_gb300", "csrc")

PROGRAM = r"""
#include "device_once.cuh"
#include <cstdio>
#include <cstdlib>
static int device = 0, calls[256], asked = 0;
static cudaError_t result = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int)
{
    ++calls[device];
    return result;
}
extern "C" cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int d) { *v = 100 + d; return cudaSuccess; }
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t)
{
    ++asked;
    *n = 2;
    return cudaSuccess;
}
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)
static void k1(int) {}
static void k2(float) {}
int main()
{
    sparc::DeviceOnce a, n;
    for (int rep = 0; rep < 3; ++rep)                      // every device is set once
        for (device = 0; device < 3; ++device) CHECK(a.allow_smem(1 << 16, k1, k2) == cudaSuccess);
    for (int d = 0; d < 3; ++d) CHECK(calls[d] == 2);
    device = 5;                                            // a failure is not kept
    result = cudaErrorInvalidValue;
    CHECK(a.allow_smem(1 << 16, k1, k2) == cudaErrorInvalidValue && calls[5] == 1);
    result = cudaSuccess;
    CHECK(a.allow_smem(1 << 16, k1, k2) == cudaSuccess && calls[5] == 3);
    CHECK(a.allow_smem(1 << 16, k1, k2) == cudaSuccess && calls[5] == 3);
    device = 200;                                          // beyond the table: asked each time
    CHECK(a.allow_smem(1 << 16, k1) == cudaSuccess && a.allow_smem(1 << 16, k1) == cudaSuccess);
    CHECK(calls[200] == 2);
    for (int rep = 0; rep < 2; ++rep)                      // values differ by device
        for (device = 0; device < 4; ++device) {
            int v = 0;
            auto ask = [](int dev, int &m) { return sparc::coop_blocks((const void *)k1, 256, dev, m); };
            CHECK(n.get(v, ask) == cudaSuccess && v == 2 * (100 + device));
        }
    CHECK(asked == 4);
    return 0;
}
"""


def test_kept_per_device(tmp_path):
    cxx = shutil.which("g++")
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-x", "c++", "-I", CSRC, "-I", inc, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_attributes_are_set_nowhere_else():
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        if os.path.basename(f) == "device_once.cuh":
            continue
        text = open(f).read()
        for call in ("cudaFuncSetAttribute", "cudaOccupancyMaxActiveBlocksPerMultiprocessor"):
            assert call not in text, (os.path.basename(f), call)
        # no process-wide cache of a device's property
        assert not re.search(r"static std::atomic<(bool|int)>", text), os.path.basename(f)
