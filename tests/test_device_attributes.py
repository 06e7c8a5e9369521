"""Kernel attributes are set once per device, not once per process (no GPU).

once_per_device is compiled for the host against a stand-in for cudaGetDevice; the sources are checked
to set kernel attributes either through it or on every call.
"""
import glob
import os
import re
import shutil
import subprocess

import pytest

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300")
CSRC = os.path.join(PKG, "csrc")

PROGRAM = r"""
#include "mppi_internal.h"
#include <stdio.h>
static int device = 0;
static cudaError_t device_error = cudaSuccess;
extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = device; return device_error; }
#define EXPECT(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    std::atomic<unsigned long long> done{0};
    int calls = 0, last = -1;
    cudaError_t result = cudaSuccess;
    auto set = [&](int dev) { ++calls; last = dev; return result; };
    for (int d : {0, 1, 63}) {
        device = d;
        EXPECT(mppi::once_per_device(done, set) == cudaSuccess && last == d);
    }
    EXPECT(calls == 3);
    for (int d : {63, 0, 1, 0}) {
        device = d;
        EXPECT(mppi::once_per_device(done, set) == cudaSuccess);
    }
    EXPECT(calls == 3);
    device = 2;                       // a failure is reported and tried again
    result = cudaErrorInvalidValue;
    EXPECT(mppi::once_per_device(done, set) == cudaErrorInvalidValue && calls == 4);
    result = cudaSuccess;
    EXPECT(mppi::once_per_device(done, set) == cudaSuccess && calls == 5);
    EXPECT(mppi::once_per_device(done, set) == cudaSuccess && calls == 5);
    device = 64;                      // past the last bit: each time
    EXPECT(mppi::once_per_device(done, set) == cudaSuccess && calls == 6 && last == 64);
    EXPECT(mppi::once_per_device(done, set) == cudaSuccess && calls == 7);
    device_error = cudaErrorNoDevice;
    EXPECT(mppi::once_per_device(done, set) == cudaErrorNoDevice && calls == 7);
    return 0;
}
"""


def test_each_device_is_set_once(tmp_path):
    from paper_2308_01654_gb300 import _build
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", include, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_kernel_attribute_is_remembered_for_the_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        assert not re.search(r"static\s+(std::atomic<bool>|bool|std::once_flag)\s+done", text), path
        for m in re.finditer(r"cudaFuncSetAttribute", text):
            before = text[:m.start()]
            body = before[before.rindex("\nstatic "):]                 # the function that sets it
            assert "once_per_device" in body or "static std::" not in body, path
