"""The integer FP64 <-> FP32 conversions of the layout passes (csrc/convert.cuh),
built for the host: bit-identical to the casts wherever they claim the value,
over exponents at both ends of the FP32 range, ties, carries and zeros, and
every infinity, NaN, subnormal and out-of-range value is handed back."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <stddef.h>
#include "convert.cuh"
extern "C" void d2f(const uint64_t* d, uint32_t* f, uint8_t* other, size_t n) {
  for (size_t i = 0; i < n; ++i) {
    bool o = false;
    f[i] = mglma::d2f_bits((uint32_t)(d[i] >> 32), (uint32_t)d[i], o);
    other[i] = o;
  }
}
extern "C" void f2d(const uint32_t* f, uint64_t* d, uint8_t* other, size_t n) {
  for (size_t i = 0; i < n; ++i) {
    bool o = false;
    uint32_t hi, lo;
    mglma::f2d_bits(f[i], hi, lo, o);
    d[i] = ((uint64_t)hi << 32) | lo;
    other[i] = o;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import ctypes
    d = tmp_path_factory.mktemp("cvt")
    (d / "c.cc").write_text(SRC)
    so = d / "c.so"
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2412_06347_gb300", "csrc"),
                    str(d / "c.cc"), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def call(lib, name, x, out_dtype):
    import ctypes
    y, o = np.empty(x.size, out_dtype), np.empty(x.size, np.uint8)
    getattr(lib, name)(x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p),
                       o.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(x.size))
    return y, o.astype(bool)


def test_double_to_float(lib):
    rng = np.random.default_rng(5)
    exps = np.array([0, 1, 870, 872, 895, 896, 897, 898, 1000, 1023, 1149, 1150, 1151, 1152, 2046, 2047], np.uint64)
    low29 = np.array([0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1], np.uint64)
    top23 = np.concatenate([np.array([0, 1, 2, (1 << 23) - 2, (1 << 23) - 1]), rng.integers(0, 1 << 23, 40)]).astype(np.uint64)
    g = np.array(np.meshgrid(exps, top23, low29, np.array([0, 1], np.uint64), indexing="ij")).reshape(4, -1)
    x = (g[3] << np.uint64(63)) | (g[0] << np.uint64(52)) | (g[1] << np.uint64(29)) | g[2]
    x = np.ascontiguousarray(np.concatenate([x, rng.integers(0, 1 << 63, 200000).astype(np.uint64)]))
    f, other = call(lib, "d2f", x, np.uint32)
    d = x.view(np.float64)
    with np.errstate(all="ignore"):
        want = d.astype(np.float32)
    assert np.array_equal(f[~other], want.view(np.uint32)[~other])
    e = (x >> np.uint64(52)) & np.uint64(2047)
    zero = (x << np.uint64(1)) == 0
    assert np.array_equal(other, ~(zero | ((e >= 897) & (e <= 1150))))


def test_float_to_double(lib):
    rng = np.random.default_rng(6)
    x = np.concatenate([np.array([0, 1, 0x007fffff, 0x00800000, 0x7f7fffff, 0x7f800000, 0x7fc00000, 0x3f800000]),
                        rng.integers(0, 1 << 31, 200000)]).astype(np.uint32)
    x = np.ascontiguousarray(np.concatenate([x, x | np.uint32(0x80000000)]))
    d, other = call(lib, "f2d", x, np.uint64)
    with np.errstate(all="ignore"):
        want = x.view(np.float32).astype(np.float64)
    assert np.array_equal(d[~other], want.view(np.uint64)[~other])
    e = (x >> np.uint32(23)) & np.uint32(255)
    zero = (x << np.uint32(1)) == 0
    assert np.array_equal(other, ~(zero | ((e >= 1) & (e <= 254))))
