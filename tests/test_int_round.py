"""oz_i64x2_round(hi, lo, w, p), the fitting GEMMs' conversion of a group sum
(oz.cuh): the double nearest (ties to even) to (hi 2^w + lo) 2^p, compiled for
the host from the header and checked against exact rational arithmetic."""
import ctypes
import os
import random
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "oz.cuh"
extern "C" double t_round(long long hi, long long lo, int w, int p) { return oz_i64x2_round(hi, lo, w, p); }
'''


@pytest.fixture(scope="module")
def t_round(tmp_path_factory):
    d = tmp_path_factory.mktemp("ozround")
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I",
                        os.path.join(ROOT, "paper_2004_11658_gb300", "csrc"), "-I", "/usr/local/cuda/include", str(src),
                        "-o", str(so)], capture_output=True, text=True)
    if r.returncode != 0:
        pytest.skip("host compiler or CUDA headers unavailable: " + r.stderr[-300:])
    f = ctypes.CDLL(str(so)).t_round
    f.restype = ctypes.c_double
    f.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return f


@pytest.mark.parametrize("w", [12, 14, 28, 32])   # beta (S - H) of the digit plans, and the widest
def test_nearest_even(t_round, w):
    rng = random.Random(w)
    cases = [(0, 0), (0, 1), (0, -1), (1, 0), (-1, 0), (1, -(1 << w)), (-1, 1 << w)]
    for _ in range(20000):
        hi = rng.randrange(1 << rng.randrange(0, 61)) * rng.choice((1, -1))
        lo = rng.randrange(1 << rng.randrange(0, 60)) * rng.choice((1, -1))
        cases.append((hi, lo))
    # ties and their neighbours: 53 kept bits, a half, and one unit either side
    for _ in range(5000):
        m = rng.randrange(1 << 52, 1 << 53)
        e = rng.randrange(1, w + 8)
        X = ((2 * m + 1) << (e - 1)) + rng.choice((-1, 0, 0, 1))
        X *= rng.choice((1, -1))
        lo = X % (1 << w) + rng.choice((0, 1, -1)) * (1 << w)
        cases.append(((X - lo) >> w, lo))
    for hi, lo in cases:
        p = rng.randrange(-300, 300)
        X = Fraction(hi) * 2 ** w + lo
        ref = float(X * Fraction(2) ** p)   # correctly rounded, ties to even
        assert t_round(hi, lo, w, p) == ref, (hi, lo, w, p)
