// residual_sum.h -- one entry of the J-orthogonality residual of a pivot's V, by integer operations.
//
// M_xj = 2^E (hi 2^28 + lo) + x + y in FP32: a digit product of at most 64 terms (|hi| < 5 2^37,
// |lo| < 2^43) and the two linear terms.  The terms are aligned to a common unit of 2^-55 of the largest
// possible product of two entries or 2^-58 of x and y, each rounded to nearest, so the sum is as accurate as
// an FP64 one and as free of bias: M drives V to J-unitarity, so what it is always off by stays in V and
// adds up over the steps (with the low bits cut off |V^T J V - J| came out 1.3 times as large).
// GB300 issues ~1.6 FP64 operations per clock per SM; the FP64 form took 7 per entry, ~9k clocks per
// residual of a 64-column block.
// Host and device code (the host side serves the CPU tests of this arithmetic).
#pragma once
#include "oz_assemble.h"

namespace jac {

OZ_HD unsigned long long oz_double_bits(double x) {
#if defined(__CUDA_ARCH__)
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long b;
  memcpy(&b, &x, sizeof(b));
  return b;
#endif
}
OZ_HD float oz_pow2f(int e) {  // -126 <= e <= 127
#if defined(__CUDA_ARCH__)
  return __int_as_float((e + 127) << 23);
#else
  const unsigned b = (unsigned)(e + 127) << 23;
  float f;
  memcpy(&f, &b, sizeof(f));
  return f;
#endif
}
OZ_HD int oz_clamp_i(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }
OZ_HD unsigned oz_min_u(unsigned a, unsigned b) { return a < b ? a : b; }

// x in units of 2^(ub - 1075), to nearest; ub >= (biased exponent of x) - 6
OZ_HD long long oz_align(double x, int ub) {
  const unsigned long long u = oz_double_bits(x);
  const int e = (int)((u >> 52) & 0x7ff);
  unsigned long long m = ((u & ((1ull << 52) - 1)) | (e ? 1ull << 52 : 0ull)) << 7;
  m = ((m >> oz_min_u((unsigned)(ub + 6 - (e ? e : 1)), 62u)) + 1) >> 1;
  return (u >> 63) ? -(long long)m : (long long)m;
}

OZ_HD float oz_residual_entry(long long hi, long long lo, int E, double x, double y) {
  const int ex = (int)((oz_double_bits(x) >> 52) & 0x7ff), ey = (int)((oz_double_bits(y) >> 52) & 0x7ff);
  const int emax = ex > ey ? ex : ey, ulin = (emax ? emax : 1) - 6;
  // units of 2^(ub - 1075): hi 2^28 + lo = (hi 2^22 + (lo >> 6)) 2^6, so its unit is 2^(E + 6)
  const int up = E + 6 + 1075, ub = ulin > up ? ulin : up;
  const long long q = (hi << 22) + ((lo + 32) >> 6);  // |q| < 2^62
  const long long s = ((((2 * q) >> oz_min_u((unsigned)(ub - up), 62u)) + 1) >> 1) + oz_align(x, ub) + oz_align(y, ub);
  const int sh = ub - 1075;  // s 2^sh, in two exact steps (FP32 range)
  const int h = oz_clamp_i(sh / 2, -120, 120), h2 = oz_clamp_i(sh - h, -120, 120);
  return ((float)s * oz_pow2f(h)) * oz_pow2f(h2);
}

}  // namespace jac
