"""oz_digit_at(I + oz_digit_bias) against oz_digit_step's carry chain (oz.cuh):
the same balanced digits, read from their places, compiled for the host from the
header, over random integers, the largest ones and runs of the tie digit."""
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
    for (int sd = S - 1; sd >= 0; --sd)
        if (oz_digit_at(J, S, beta, sd) != (sd > 0 ? oz_digit_step(I, beta) : (int)I)) return sd + 1;
    return 0;
}
'''


@pytest.fixture(scope="module")
def t_cmp(tmp_path_factory):
    d = tmp_path_factory.mktemp("ozdigit")
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I",
                        os.path.join(ROOT, "paper_2004_11658_gb300", "csrc"), "-I", "/usr/local/cuda/include", str(src),
                        "-o", str(so)], capture_output=True, text=True)
    if r.returncode != 0:
        pytest.skip("host compiler or CUDA headers unavailable: " + r.stderr[-300:])
    f = ctypes.CDLL(str(so)).t_cmp
    f.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return f


@pytest.mark.parametrize("S,beta", [(8, 7), (4, 7), (5, 6)])
def test_same_digits(t_cmp, S, beta):
    rng = random.Random(S)
    top = 1 << (beta * S)                       # |x| 2^(beta S - e) <= 2^(beta S)
    half = 1 << (beta - 1)
    cases = [0, 1, -1, top, -top, top - 1, 1 - top]
    for _ in range(50000):
        cases.append(rng.randrange(1 << rng.randrange(1, beta * S + 1)) * rng.choice((1, -1)))
    for _ in range(5000):                       # digits at, and one off, the tie
        cases.append(sum((half + rng.choice((-1, 0, 1))) << (beta * q) for q in range(rng.randrange(1, S)))
                     * rng.choice((1, -1)))
    for I in cases:
        assert t_cmp(I, S, beta) == 0, (I, S, beta)
