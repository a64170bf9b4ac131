"""oz_assemble_small (csrc/oz_assemble.h) on the CPU: the double nearest to 2^e (hi 2^sh + lo), bit for
bit, in the ranges of the digit kernels (sh = 28 and 35) and at the limits of its own."""
import ctypes
import math
import os
import random
import struct
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "oz_assemble.h"
extern "C" double assemble(long long hi, long long lo, int sh, int e) { return jac::oz_assemble_small(hi, lo, sh, e); }
extern "C" double general(long long hi, long long lo, int sh, int e) { return jac::oz_assemble(hi, lo, sh, e); }
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("assemble")
    cpp, so = d / "a.cpp", d / "a.so"
    cpp.write_text(SRC)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++14", "-shared", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_1008_0201_gb300", "csrc"), "-o", str(so), str(cpp)], check=True)
    L = ctypes.CDLL(str(so))
    for f in (L.assemble, L.general):
        f.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
        f.restype = ctypes.c_double
    return L


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def check(lib, hi, lo, sh, e):
    s = (hi << sh) + lo
    want = math.ldexp(float(s), e) if s else 0.0
    assert bits(lib.assemble(hi, lo, sh, e)) == bits(want) == bits(lib.general(hi, lo, sh, e)), (hi, lo, sh, e)


@pytest.mark.parametrize("sh,hb,lb", [(28, 51, 51), (35, 43, 50), (28, 62, 62), (35, 62, 62), (1, 62, 62), (40, 61, 62)])
def test_random_and_adversarial(lib, sh, hb, lb):
    g = random.Random(sh * 100 + hb)
    for _ in range(20000):
        h = g.randrange(-(2 ** g.randrange(1, hb)), 2 ** g.randrange(1, hb))
        l = g.randrange(-(2 ** g.randrange(1, lb)), 2 ** g.randrange(1, lb))
        check(lib, h, l, sh, g.randrange(-200, 200))
    for p in range(0, min(hb + sh, 100)):  # ties and their neighbours around every size of the sum
        for d in (-1, 0, 1):
            for odd in (0, 1):
                s = (2 ** p) * 2 + (2 ** max(p - 52, 0)) * odd + 2 ** max(p - 53, 0) + d
                for sg in (1, -1):
                    h, l = (sg * s) >> sh, (sg * s) & (2 ** sh - 1)
                    if abs(h) < 2 ** hb:
                        check(lib, h, l, sh, 0)
                        check(lib, h, l, sh, -90)


@pytest.mark.parametrize("e", [-1100, -1085, -1074, 960, 900])
def test_limits_of_the_exponent(lib, e):
    g = random.Random(5)
    for h, l in [(0, 0), (1, 0), (-1, 0), (0, 1), (2 ** 40, -1), (-(2 ** 40), 1), (1, -(2 ** 28))] + [
            (g.randrange(-2 ** 40, 2 ** 40), g.randrange(-2 ** 40, 2 ** 40)) for _ in range(200)]:
        assert bits(lib.assemble(h, l, 28, e)) == bits(lib.general(h, l, 28, e))
