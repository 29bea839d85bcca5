"""f2d and d2f (conv.cuh), the mixed kernels' conversions, against the casts, bit for
bit: random patterns of every exponent, ties and their neighbours, carries into
the exponent, the ends of the normal FP32 range, zeros, subnormals, infinities;
NaN stays NaN.  Compiled for the host from the header."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "conv.cuh"
extern "C" void t_f2d(const float *x, double *y, long n) { for (long i = 0; i < n; ++i) y[i] = f2d(x[i]); }
extern "C" void t_d2f(const double *x, float *y, long n) { for (long i = 0; i < n; ++i) y[i] = d2f(x[i]); }
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("conv")
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I",
                        os.path.join(ROOT, "paper_2004_11658_gb300", "csrc"), "-I", "/usr/local/cuda/include", str(src),
                        "-o", str(so)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-500:]
    return ctypes.CDLL(str(so))


def call(f, x, out):
    y = np.empty(len(x), dtype=out)
    f(x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p), ctypes.c_long(len(x)))
    return y


def same(got, want, bits):
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(bits), want[~nan].view(bits))


def test_f2d(lib):
    rng = np.random.default_rng(0)
    u = rng.integers(0, 1 << 32, 2000000, dtype=np.uint64).astype(np.uint32)
    edge = np.array([(s << 31) | (e << 23) | m for s in (0, 1) for e in (0, 1, 2, 126, 127, 128, 253, 254, 255)
                     for m in (0, 1, 2, 0x400000, 0x7ffffe, 0x7fffff)], dtype=np.uint32)
    x = np.concatenate([u, edge]).view(np.float32)
    with np.errstate(invalid="ignore"):   # signalling NaN patterns
        same(call(lib.t_f2d, x, np.float64), x.astype(np.float64), np.uint64)


def test_d2f(lib):
    rng = np.random.default_rng(1)
    mant = rng.integers(0, 1 << 52, 2000000, dtype=np.uint64)
    sign = rng.integers(0, 2, len(mant), dtype=np.uint64) << np.uint64(63)
    exps = rng.integers(0, 2048, len(mant), dtype=np.uint64)
    near = rng.integers(890, 1160, len(mant), dtype=np.uint64)   # around and inside the FP32 range
    tie = (mant >> np.uint64(29) << np.uint64(29)) + np.uint64(1 << 28)
    ones = np.uint64((1 << 52) - 1) - (mant >> np.uint64(24))    # mantissas that carry
    parts = [sign | (exps << np.uint64(52)) | mant]
    for m in (mant, tie, tie + np.uint64(1), tie - np.uint64(1), ones):
        parts.append(sign | (near << np.uint64(52)) | m)
    edge = np.array([(s << 63) | (e << 52) | m for s in (0, 1)
                     for e in (0, 1, 872, 873, 874, 895, 896, 897, 898, 1149, 1150, 1151, 1152, 2046, 2047)
                     for m in (0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1, 1 << 29, 3 << 28,
                               (1 << 52) - (1 << 29), (1 << 52) - (1 << 28) - 1, (1 << 52) - (1 << 28), (1 << 52) - 1)],
                    dtype=np.uint64)
    x = np.concatenate(parts + [edge]).view(np.float64)
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        same(call(lib.t_d2f, x, np.float32), x.astype(np.float32), np.uint32)
