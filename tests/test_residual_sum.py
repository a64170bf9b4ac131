"""One entry of the pivot's J-orthogonality residual (csrc/residual_sum.h), compiled for the host, against
exact integers: M = 2^E (hi 2^28 + lo) + x + y.

Each of the three terms is rounded to nearest in one unit, so the sum is within 1.5 units (and an FP32
ulp, 2^-149 at least) of the exact value, and without bias: over n random entries the mean error stays within five
standard deviations of zero, at most 5 sqrt(3 / 12 / n) units.  The unit is 2^(E + 6), or 2^-58 of the
larger of x and y.
"""
import ctypes
import math
import os
import random
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "residual_sum.h"
extern "C" float entry(long long hi, long long lo, int E, double x, double y) {
  return jac::oz_residual_entry(hi, lo, E, x, y);
}
'''


@pytest.fixture(scope="module")
def entry(tmp_path_factory):
    d = tmp_path_factory.mktemp("res")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1008_0201_gb300", "csrc"), "-o", str(d / "r.so"), str(d / "r.cpp")], check=True)
    fn = ctypes.CDLL(str(d / "r.so")).entry
    fn.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_double, ctypes.c_double]
    fn.restype = ctypes.c_float
    return fn


def pow2(e):
    return Fraction(2) ** e


@pytest.mark.parametrize("E", [-57, -97, -220, 0, 60])
@pytest.mark.parametrize("kind", ["cancel", "diagonal", "linear", "product"])
def test_residual_entry(entry, E, kind):
    g = random.Random(7 * E + len(kind))
    n, total = 4000, Fraction(0)
    for _ in range(n):
        big = 2 ** g.randrange(8, 42)
        big = min(big, 5 * 2 ** 37 - 1)  # 64 products of the largest digits, all levels
        hi, lo = g.randrange(-big, big + 1), g.randrange(-2 ** 42, 2 ** 42)
        if kind == "diagonal":  # a sum of squares
            hi = abs(hi)
        prod = (hi * 2 ** 28 + lo) * pow2(E)
        x, y = (math.ldexp(g.uniform(-1, 1), E + g.randrange(20, 66)) for _ in range(2))
        if kind == "cancel":  # what is left of a converged V: the linear terms undo the product
            x = float(-prod) - y if hi else x
        elif kind == "diagonal":
            x = y = float(-prod / 2)
        elif kind == "linear":
            hi = lo = 0
            prod = Fraction(0)
        elif kind == "product":
            x = y = 0.0
        got = entry(hi, lo, E, x, y)
        want = prod + Fraction(x) + Fraction(y)
        lin = max(abs(x), abs(y))
        unit = max(pow2(E + 6), pow2(math.frexp(lin)[1] - 1 - 58) if lin else Fraction(0))
        ulp = pow2(math.frexp(float(want))[1] - 24) if want else Fraction(0)
        err = Fraction(got) - want
        assert abs(err) <= Fraction(3, 2) * unit + ulp + pow2(-149), (hi, lo, E, x, y, got, float(want), float(err / unit))
        if 2 ** -120 < abs(want) < 2 ** 20 * unit:  # FP32's own rounding below 2^-4 units
            total += err / unit
    assert abs(float(total)) <= 5.0 * math.sqrt(n * 3 / 12.0)
