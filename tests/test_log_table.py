"""The sampler's FP64 logarithm (csrc/log_device.cuh), compiled for the host with
the few intrinsics that it names: the alignment that its 16-byte loads need, and its
error against a wider logarithm over the arguments that the sampler has."""
import ctypes
import os
import subprocess

import numpy as np
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


def ulps(log_lib, x):
    """|log_pos(x) - log x| in units of the result's last place; log x in the platform's
    long double (64 bits of mantissa or more: 2^-11 of such a unit)."""
    x = np.ascontiguousarray(x, np.float64)
    y = np.empty_like(x)
    ptr = ctypes.POINTER(ctypes.c_double)
    log_lib.logs(x.ctypes.data_as(ptr), y.ctypes.data_as(ptr), len(x))
    want = np.log(x.astype(np.longdouble))
    unit = np.spacing(np.abs(want.astype(np.float64)))
    return np.abs((y.astype(np.longdouble) - want) / unit).astype(np.float64)


G = np.random.default_rng(11)
U = (G.integers(0, 1 << 32, 400_000).astype(np.float64) + 0.5) * 2.0 ** -32
ARGUMENTS = {
    "uniforms": U,
    "their squares": U * U,
    "half to one": G.uniform(0.5, 1.0, 400_000),
    "around one": 1.0 + G.uniform(-0.01, 0.01, 400_000),
    "roots": np.exp(G.uniform(np.log(1e-17), np.log(50.0), 400_000)),
    # the first argument of each row, the last of the row before, one either side
    "row edges": ((np.int64(0x3FE6A000) << 32) + (np.arange(129, dtype=np.int64)[:, None] << 45)
                  + np.arange(-2, 3)[None, :]).reshape(-1).view(np.float64),
    "next to one": np.concatenate([1.0 + np.arange(1, 200) * 2.0 ** -52, 1.0 - np.arange(1, 200) * 2.0 ** -53]),
    "extremes": np.array([2.0 ** -1022, 2.0 ** -1021 * 1.3, 1.7976931348623157e308, 2.0 ** 1023]),
}


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="needs a long double wider than double")
@pytest.mark.parametrize("name", list(ARGUMENTS))
def test_logarithm_to_half_a_unit(log_lib, name):
    """0.5 for the last rounding and eight roundings (the products and sums of log1p's tail,
    its coefficients) of at most 2^-8: with a tabulated c the result is at least 2^-8 and
    the tail at most 2^-15; around 1 the tail is at most 2^-8 of the result."""
    assert ulps(log_lib, ARGUMENTS[name]).max() <= 0.5 + 8 * 2.0 ** -8 + 2.0 ** -11


def test_logarithm_of_one(log_lib):
    y, one = np.ones(1), np.ones(1)
    ptr = ctypes.POINTER(ctypes.c_double)
    log_lib.logs(one.ctypes.data_as(ptr), y.ctypes.data_as(ptr), 1)
    assert y[0] == 0.0
