"""The sampler's FP64 logarithm (csrc/log_device.cuh), compiled for the host with
the few intrinsics that it names: the alignment that its 16-byte loads need."""
import ctypes
import os
import subprocess

import pytest

from paper_2412_03489_gb300 import build as hb

SHIM = r"""
#include <cmath>
#include <cstring>
#include <cstdint>
#include <cuda_runtime.h>
using std::fma;
static inline int __double2hiint(double x) { uint64_t b; memcpy(&b, &x, 8); return (int)(b >> 32); }
static inline int __double2loint(double x) { uint64_t b; memcpy(&b, &x, 8); return (int)b; }
static inline double __hiloint2double(int h, int l) {
    const uint64_t b = ((uint64_t)(uint32_t)h << 32) | (uint32_t)l;
    double x; memcpy(&x, &b, 8); return x;
}
static inline double2 __ldg(const double2* p) { return *p; }
static inline double __ldg(const double* p) { return *p; }
#include "log_device.cuh"
extern "C" int table_alignment() { return (int)__alignof__(hr::kLogTable); }
extern "C" int row_bytes() { return (int)sizeof(hr::kLogTable[0]); }
extern "C" void logs(const double* x, double* y, int n) { for (int i = 0; i < n; ++i) y[i] = hr::log_pos(x[i]); }
"""


@pytest.fixture(scope="module")
def log_lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("log")
    src, out = d / "log.cpp", d / "log.so"
    src.write_text(SHIM)
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I" + cuda, "-I" + hb.CSRC,
                    str(src), "-o", str(out)], check=True, capture_output=True, text=True)
    return ctypes.CDLL(str(out))


def test_rows_are_aligned_for_their_vector_loads(log_lib):
    """A row's first two values are one 16-byte load: the table's declaration itself has
    to ask for that alignment (an array of doubles alone is aligned to 8 bytes wherever
    the compiler happens to place it; the type's alignment is what every copy has)."""
    assert log_lib.table_alignment() % 16 == 0
    assert log_lib.row_bytes() % 16 == 0
