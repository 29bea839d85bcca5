"""oz_digit_f32(I + oz_digit_bias) (oz.cuh), the digits as the kernels pack them: the
upper half of each float is the BF16 of oz_digit_step's digit and the lower half
0.  Compiled for the host from the header, over random integers, the largest ones
and runs of the tie digit."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "oz.cuh"
extern "C" int t_cmp(long long I, int S, int beta)
{
    const long long J = I + oz_digit_bias(S, beta);
    for (int sd = S - 1; sd >= 0; --sd) {
        const float f = oz_digit_f32(J, S, beta, sd);
        uint32_t u;
        std::memcpy(&u, &f, 4);
        if (u != (uint32_t)oz_bf16_int(sd > 0 ? oz_digit_step(I, beta) : (int)I) << 16) return sd + 1;
    }
    return 0;
}
'''


@pytest.fixture(scope="module")
def t_cmp(tmp_path_factory):
    d = tmp_path_factory.mktemp("ozfloat")
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I",
                        os.path.join(ROOT, "paper_2004_11658_gb300", "csrc"), "-I", "/usr/local/cuda/include", str(src),
                        "-o", str(so)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-500:]
    f = ctypes.CDLL(str(so)).t_cmp
    f.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return f


@pytest.mark.parametrize("S,beta", [(8, 7), (4, 7), (5, 6)])   # the plans of the fitting GEMMs
def test_packed_digits(t_cmp, S, beta):
    rng = random.Random(S)
    top, half = 1 << (beta * S), 1 << (beta - 1)
    cases = [0, 1, -1, top, -top, top - 1, 1 - top]
    for _ in range(50000):
        cases.append(rng.randrange(1 << rng.randrange(1, beta * S + 1)) * rng.choice((1, -1)))
    for _ in range(5000):
        cases.append(sum((half + rng.choice((-1, 0, 1))) << (beta * q) for q in range(rng.randrange(1, S)))
                     * rng.choice((1, -1)))
    for I in cases:
        assert t_cmp(I, S, beta) == 0, (I, S, beta)


def test_sums_of_a_segment_are_exact():
    """The plan of the FP64 GEMMs, 8 digits of 7 bits: the group of most products (8 or
    9 pairs: the first digit up to 2^7, the others up to 2^6) over one segment of 25
    chunks stays below 2^24, and so do the 16 chunks of a weight gradient's segment."""
    S, beta = 8, 7
    first, other = 1 << beta, 1 << (beta - 1)
    per_column = max(sum((first if s == 1 else other) * (first if g - s == 1 else other)
                         for s in range(max(1, g - S), min(S, g - 1) + 1)) for g in range(2, S + 2))
    seg = 16777215 // (4096 * 10) // 16
    assert seg == 25 and seg * 16 * per_column < 1 << 24 and 16 * 16 * per_column < 1 << 24
