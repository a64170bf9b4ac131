"""CPU model of the biased digit split (csrc/ozaki.cuh: oz_biased, oz_split2): the same balanced
digits as the carry form, in the 28-bit halves and FP16 patterns the kernels use."""
import random

import numpy as np
import pytest

from test_digit_split_model import bexp, fixed, split

BIAS = 64 * ((2 ** 56 - 1) // 127)


def biased(x, d):
    u = int(np.float64(x).view(np.uint64))
    m = ((u & (2 ** 52 - 1)) | 2 ** 52) << 3
    if ((u >> 52) & 0x7FF) == 0:
        m = 0
    sh = min((-d) & 0xFFFFFFFF, 63)
    a = ((m >> sh) + 1) >> 1
    return BIAS - a if u >> 63 else BIAS + a


def split2(v0, v1):
    w = [None] * 8
    for h in range(2):
        a, b = (v0 >> (28 * h)) & 0xFFFFFFFF, (v1 >> (28 * h)) & 0xFFFFFFFF
        for j in range(4):
            m = 0xFF if h == 1 and j == 3 else 0x7F
            hi = (b << (16 - 7 * j)) & 0xFFFFFFFF if 7 * j <= 16 else b >> (7 * j - 16)
            x = ((a >> (7 * j)) & m) | 0x64006400 | (hi & (m << 16))
            pair = np.array([x & 0xFFFF, x >> 16], dtype=np.uint16).view(np.float16)
            w[7 - 4 * h - j] = [float(p) - 1088.0 for p in pair]
    return [p[0] for p in w], [p[1] for p in w]


def values():
    r = random.Random(3)
    xs = [0.0, 5e-324, 1.0, -1.0, np.nextafter(2.0, 0), -np.nextafter(2.0, 0), 1.5, 2.0 ** -1022]
    return xs + [r.uniform(-2, 2) * 2.0 ** r.randrange(-70, 1) for _ in range(400)]


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 30, 52, 54, 55, 57, 58, 61, 62, 63, 64, 2000])
def test_biased_split_equals_balanced_split(shift):
    xs = values()
    top = bexp(1.0) + shift  # group bound at or above every value (bexp of values in [1, 2) + shift)
    for x0, x1 in zip(xs, xs[1:] + xs[:1]):
        V = [fixed(x, bexp(x) - top) for x in (x0, x1)]
        b = [biased(x, bexp(x) - top) for x in (x0, x1)]
        assert [v + BIAS for v in V] == b
        assert [list(map(float, split(v))) for v in V] == list(split2(*b))


def test_positive_exponent_of_an_empty_group_gives_zero_digits():
    # a group without nonzero entries has a bound far below any exponent: d > 0, value zero
    assert biased(0.0, 100000 - 0) == BIAS
    assert split2(BIAS, BIAS) == ([0.0] * 8, [0.0] * 8)


@pytest.mark.parametrize("V", [2 ** 55 - 1, -(2 ** 55 - 1), 2 ** 55 - 64, 64 * 128 ** 3, -64 * 128 ** 7 + 1])
def test_extreme_integers(V):
    assert list(map(float, split(V))) == split2(V + BIAS, BIAS)[0]
