"""The parameters of an inner rotation (csrc/rotation.h), compiled for the host, against FP64 over the
whole FP32 range of squared column norms.

Rounding (eps = 2^-24): the unit cancels, nu and s carry one rounding each, so trigonometric
rr = nu^2 + 4 s^2 is good to 4 eps, h to 4, nu h and s h to 6, c2 >= 1/2 to 7, 1 / cos to 5.5 and the
sine to 13 eps; hyperbolic with 2 |a_ij| <= 0.8 x rr loses 1 / 0.36 to cancellation (15 eps) and the
sine is good to 20 eps.  Results below FP32's normal range: one subnormal unit more.
"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "rotation.h"
extern "C" void angle(float aii, float ajj, float x, float b, int trig, float* out) {
  const float sg = trig ? 1.0f : -1.0f;
  const jac::RotUnit q = jac::rot_unit(aii, ajj, x);
  const jac::RotAngle r = jac::rot_angle(q, sg, 4.0f * sg, b);
  out[0] = r.c, out[1] = r.s, out[2] = r.cinv, out[3] = r.guard, out[4] = b * q.rs;
}
'''
EPS = 2.0 ** -24
COS = [0.9, 0.5, 1e-2, 1e-5, 1e-10, 1e-16, 1e-22]


@pytest.fixture(scope="module")
def angle(tmp_path_factory):
    d = tmp_path_factory.mktemp("rot")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1008_0201_gb300", "csrc"), "-o", str(d / "r.so"), str(d / "r.cpp")], check=True)
    fn = ctypes.CDLL(str(d / "r.so")).angle
    fn.argtypes = [ctypes.c_float] * 4 + [ctypes.c_int, ctypes.c_void_p]
    out = np.zeros(5, dtype=np.float32)

    def call(aii, ajj, x, b, trig):
        fn(float(aii), float(ajj), float(x), float(b), int(trig), out.ctypes.data)
        return [float(v) for v in out]

    return call


@pytest.mark.parametrize("trig", [True, False])
@pytest.mark.parametrize("ratio", [1.0, 1.0 + 1e-6, 3.0, 1e6, 1e12, 1e17, 1e18, 2e18, 1e21, 1e24, 1e30, 1e36, 1e60])
def test_angle_over_the_fp32_range(angle, ratio, trig):
    f = np.float32
    seen = 0
    for mid in 10.0 ** np.arange(-44.0, 38.0, 1.0):
        with np.errstate(over="ignore", under="ignore"):
            big, small = f(mid * math.sqrt(ratio)), f(mid / math.sqrt(ratio))
        if not (1e-44 <= small and big <= 1e37):
            continue
        for aii, ajj in ((big, small), (small, big)):
            with np.errstate(under="ignore"):
                x = f(ajj - aii) if trig else f(aii + ajj)
            for cos in COS:
                b = f(cos * math.sqrt(float(aii) * float(ajj)))
                if b == 0 or (not trig and 2 * float(b) > 0.8 * float(x)):
                    continue
                c, s, cinv, guard, _ = angle(aii, ajj, abs(x) if not trig else x, b, trig)
                if trig:
                    phi = 0.5 * math.atan2(2 * float(b), abs(float(x)))
                    want_s, want_c, tol = math.sin(phi), math.cos(phi), 13 * EPS
                else:
                    phi = 0.5 * math.atanh(2 * float(b) / float(x))
                    want_s, want_c, tol = math.sinh(phi), math.cosh(phi), 20 * EPS
                at = (ratio, mid, cos, aii, ajj, x, b)
                assert not guard, at
                assert abs(s - want_s) <= tol * want_s + 2.0 ** -149, (at, s, want_s)
                assert abs(c - want_c) <= tol * want_c, (at, c, want_c)
                assert abs(c * cinv - 1.0) <= tol, at
                seen += 1
    assert seen > 20


def test_hyperbolic_guard(angle):
    # 2 |a_ij| >= x by rounding: tanh = 0.9 whatever the size of the norms
    for a in (1e-40, 1e-30, 1.0, 1e30, 1e37):
        a = float(np.float32(a))
        c, s, _, guard, _ = angle(a, a, 2 * a, a, False)
        assert guard and abs(s / c - 0.9) < 1e-6 and abs(c * c - s * s - 1.0) < 1e-6
