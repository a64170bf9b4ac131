// rotation.h -- parameters of one pointwise rotation of the inner sweep (pivot.cu), in FP32.
//
// For two columns with squared norms a_ii, a_jj and x = a_jj - a_ii (trigonometric, Eq. (2.1):
// cot(2 phi) = x / (2 |a_ij|)) or x = a_ii + a_jj (hyperbolic: coth(2 phi) = -x / (2 |a_ij|)), with
// everything multiplied by a unit u > 0 (nu = |x| u, s = |a_ij| u):
//   h = 1 / sqrt(nu^2 +- 4 s^2),  cos(h)^2 phi = 1/2 + nu h / 2,  |sin(h) phi| = s h / cos(h) phi.
// The roots need FP32 accuracy only: the rotation is orthogonal (J-orthogonal) to their rounding
// whatever the angle.  Two MUFU operations deep after a_ij, ~90 clocks; by way of the tangent, with x
// and a_ij scaled by powers of two once both are known, it took 330.
//
// The unit is 2^30 / sqrt(a_ii a_jj) (exact against s / 2^30, the scaled entry), or about 2^62 / |x| if
// that is less, 2^126 at most: nu, s and their squares stay inside FP32's range for all norms it holds.
// It depends on the norms only and is formed beside the dot product, in four integer operations (with a
// reciprocal and float minima order 512, weight ordering, took 24.6 ms, not 24.3).
// (A nu clamped to FP32's range would set the angle: two columns whose norms differ by 1e18 would
// push each other back and forth and never settle.)
// Host and device code (the host side serves the CPU tests of this arithmetic).
#pragma once

#if defined(__CUDACC__)
#define ROT_HD __host__ __device__ __forceinline__
#else
#define ROT_HD inline
#endif
#if !defined(__CUDA_ARCH__)
#include <math.h>
#include <string.h>
#endif

namespace jac {

ROT_HD unsigned rot_bits(float x) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(x);
#else
  unsigned b;
  memcpy(&b, &x, sizeof(b));
  return b;
#endif
}
ROT_HD float rot_float(unsigned b) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(b);
#else
  float x;
  memcpy(&x, &b, sizeof(x));
  return x;
#endif
}
ROT_HD float rot_rsqrt(float x) {
#if defined(__CUDA_ARCH__)
  return rsqrtf(x);
#else
  return 1.0f / sqrtf(x);
#endif
}
// arguments of FP32 normal size
ROT_HD float rot_rsqrt_ftz(float x) {
#if defined(__CUDA_ARCH__)
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / sqrtf(x < 1.17549435e-38f ? 0.0f : x);
#endif
}

// What does not depend on a_ij: |a_ij| rs is the scaled entry, |a_ij| u and nu set the angle.
struct RotUnit {
  float rs, u, nu;
};
ROT_HD RotUnit rot_unit(float aii, float ajj, float x) {
  RotUnit q;
  q.rs = rot_rsqrt(aii) * rot_rsqrt(ajj);
  const float ax = fabsf(x);
  // positive floats order as their bits: 2^30 rs by its exponent, and 2^62 / |x| to 12% by a subtraction
  // from 2 * 127 + 62 (2^-66 at least); a value above 2^126, an infinity or a NaN loses
  const unsigned a = rot_bits(q.rs) + (30u << 23), b = (316u << 23) - rot_bits(ax);
  const unsigned m = a < b ? a : b;
  q.u = rot_float(m < 0x7e800000u ? m : 0x7e800000u);
  q.nu = ax * q.u;
  return q;
}

struct RotAngle {
  float c, s, cinv;  // cos(h) phi, |sin(h) phi|, 1 / cos(h) phi
  bool guard;        // no hyperbolic angle annihilates a_ij (2 |a_ij| >= x by rounding): tanh = 0.9, Sec. 3.2
};
// sg = 1 trigonometric, -1 hyperbolic; sg4 = 4 sg; b = |a_ij|
ROT_HD RotAngle rot_angle(const RotUnit& q, float sg, float sg4, float b) {
  RotAngle r;
  const float s = b * q.u, rr = fmaf(sg4, s * s, q.nu * q.nu);
  const float h = rot_rsqrt_ftz(rr), wh = s * h;
  const float c2 = fmaf(0.5f * q.nu, h, 0.5f);
  r.cinv = rot_rsqrt_ftz(c2);
  r.s = wh * r.cinv;
  r.c = c2 * r.cinv;
  // the cosine of a small angle as 1 -+ s^2 / 2 rounded once (rsqrt returns the value below 1 too
  // often there, and thousands of tiny rotations would shrink V: with it alone the FP32-only
  // eigenvalues of order 128 came out 5e-5 small, with this rule 2e-5)
  const float y = r.s * r.s;
  if (y < 3.8146973e-6f) r.c = fmaf(-0.5f * sg, y, 1.0f);
  r.guard = !(rr > 0.0f);
  if (r.guard) {
    r.c = 2.2941573f;
    r.s = 2.0647416f;
  }
  return r;
}

}  // namespace jac
