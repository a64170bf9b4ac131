// ozaki.cuh -- FP64-accurate products from exact FP16 tensor-core products (error-free splitting
// after Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by
// using fast routines of matrix multiplication and its applications", Numer. Algorithms 2012).
//
// GB300 runs FP16 mma.sync (FP32 accumulate) ~600x faster than FP64 mma, so the FP64 contractions
// of a step -- the Gram block A_P = G_P^* G_P (Eq. (3.4)), the update G_P V_P (Algorithm 3.4) and
// the J-orthogonality residual of V_P -- are formed from small-integer products:
//   - every value of a scale group (the entries that share one row of A or one column of B of a
//     product A B, so that the scale factors out of the contraction) is written as an integer
//     V = round(x 2^(55 - e)), |V| < 2^55, where 2^e bounds |x| over the group;
//   - V = sum_t d_t 128^(7 - t), t = 0..7, with balanced digits d_1..d_7 in [-64, 63] and
//     d_0 in [-64, 64]: every digit is an FP16 integer;
//   - digit products |d_t d_u| <= 2^12 are exact in FP16 x FP16 -> FP32, and the level sums
//     acc_L = sum over the contraction of sum_{t+u=L} d_t d_u (at most 8 products per term) stay
//     below 2^23 for up to 256 terms, where the tensor-core FP32 accumulation is exact;
//   - levels L = 0..NL-1 are kept: NL = 8 drops at most 7 * 2^-56 of the product of the two
//     group bounds per term, NL = 9 at most 6 * 2^-63;
//   - x . y = 2^(e + e' - 110) sum_L 2^(98 - 7 L) acc_L, summed in FP64.
// So each product is exact to 2^-53 of (row bound of A) x (column bound of B) per term, the
// scale of FP64 rounding itself, and the sum over levels rounds once more in FP64.
#pragma once
#include <cuda_fp16.h>

#include "oz_assemble.h"

namespace jac {

#define OZ_T 8  // digits per value

// biased exponent of |x| (0 for zero and subnormals, which the splitting treats as zero)
__device__ __forceinline__ int oz_bexp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff); }

// The split works on biased integers: V + OZ_BIAS, OZ_BIAS = sum_t 64 128^t, has the nonnegative
// base-128 fields d_t + 64, so the balanced digits need no carries, and a field becomes an FP16
// integer without a conversion instruction (16 per clock per SM on GB300): the bits 0x6400 + u are
// the half 1024 + u, and 1088 is subtracted from two at once: ~20 instructions per value instead
// of ~90 with carries and eight conversions.  With the joins of oz_value: k_gram_oz on 32 pairs of
// 2304 rows 137 -> 112 us, k_update_oz_tc there 76 -> 67 us, the adjoint of 256 problems of order
// 256 8.58 -> 6.62 ms; results bit-identical.
constexpr unsigned long long OZ_BIAS = 64ull * (((1ull << 56) - 1) / 127);

// x with biased exponent ex = oz_bexp(x) as the integer V = round(m 2^(d + 2)), m the 53-bit
// significand of |x| with its sign, for d = ex - (group bound exponent) <= 0: |V| < 2^55.  Returns
// V + OZ_BIAS.  Zeros and subnormals give V = 0 for any d.
__device__ __forceinline__ unsigned long long oz_biased(double x, int d) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  unsigned long long m = ((u & ((1ull << 52) - 1)) | (1ull << 52)) << 3;
  if (((u >> 52) & 0x7ff) == 0) m = 0;
  const unsigned sh = min((unsigned)(-d), 63u);
  const unsigned long long a = ((m >> sh) + 1) >> 1;  // round half up of m 2^(d + 2)
  return (u >> 63) ? OZ_BIAS - a : OZ_BIAS + a;
}

// The 8 digits, most significant first, of two biased integers: w[t] = (digit t of v0, of v1) as
// two FP16 integers.
__device__ __forceinline__ void oz_split2(unsigned long long v0, unsigned long long v1, unsigned (&w)[OZ_T]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // 28-bit halves: digits 7..4, then 3..0
    const unsigned a = (unsigned)(v0 >> (28 * h)), b = (unsigned)(v1 >> (28 * h));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned m = (h == 1 && j == 3) ? 0xffu : 0x7fu;  // d_0 + 64 reaches 128
      const unsigned hi = (7 * j <= 16) ? b << (16 - 7 * j) : b >> (7 * j - 16);
      const unsigned x = (((a >> (7 * j)) & m) | 0x64006400u) | (hi & (m << 16));
      __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&x), __half2half2(__ushort_as_half(0x6440)));
      w[7 - 4 * h - j] = *reinterpret_cast<unsigned*>(&r);
    }
  }
}

// D += A B, m16n8k16, FP16 operands, FP32 accumulate (no side effect: the compiler may move it)
__device__ __forceinline__ void oz_mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// four 8 x 8 FP16 matrices from shared memory; lane l gives the address of row (l & 7) of
// matrix l >> 3
__device__ __forceinline__ void oz_ldsm4(unsigned (&r)[4], const __half* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

__device__ __forceinline__ void oz_ldsm2(unsigned& r0, unsigned& r1, const __half* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(a));
}

// The digit products of one 16 x 16 (A) by 16 x 8 (B) piece into the level accumulators
// L = 0..NL-1 (NL = 8: 36 products; NL = 9: 43).  Digit t of A goes to all its levels before digit
// t + 1: two products of one level are then up to NL products apart, and the warp does not wait
// for the mma it has just issued.  (Level by level, every product waited for the one before it.)
// The sums are exact integers, so the order does not change them.
template <int NL>
__device__ __forceinline__ void oz_levels(float (&acc)[NL][4], const unsigned (&fa)[OZ_T][4],
                                          const unsigned (&fb)[OZ_T][2]) {
#pragma unroll
  for (int t = 0; t < OZ_T; ++t)
#pragma unroll
    for (int L = t; L < (t + OZ_T < NL ? t + OZ_T : NL); ++L) oz_mma(acc[L], fa[t], fb[L - t][0], fb[L - t][1]);
}

// GB300 issues ~1.6 FP64 operations per clock per SM (FP32: 128), so the recombination takes none:
// the integer level sums are gathered exactly in two int64 (hi: L = 0..3 in units of level 3, lo: L =
// 4..NL-1 in units of level NL-1, both below 2^52 for level sums below 2^23) and rounded once to
// double by integer instructions (oz_assemble_small).

// an FP32 value that holds an integer of magnitude <= 2^22, as that integer (one FP32 add: the
// integer lands in the low mantissa bits of 1.5 * 2^23 + x)
__device__ __forceinline__ int f32_small_int(float x) { return __float_as_int(x + 12582912.0f) - 0x4B400000; }

// 2^E sum_L acc_L 2^(-7 L), the acc_L exact integers held in FP32, |acc_L| <= 2^22 (up to 128 terms);
// two levels are joined in 32 bits, and the exact sum is rounded once
__device__ __forceinline__ double oz_value_int(const float (&acc)[8][4], int v, int E) {
  int q[8];
#pragma unroll
  for (int L = 0; L < 8; ++L) q[L] = f32_small_int(acc[L][v]);
  const long long hi = (long long)(q[0] * 128 + q[1]) * 16384 + (q[2] * 128 + q[3]);
  const long long lo = (long long)(q[4] * 128 + q[5]) * 16384 + (q[6] * 128 + q[7]);
  return oz_assemble_small(hi, lo, 28, E - 49);
}

// The same for nine levels and |acc_L| <= 2^23 (256 terms)
__device__ __forceinline__ double oz_value9(const float (&acc)[9][4], int v, int E) {
  int q[9];
#pragma unroll
  for (int L = 0; L < 9; ++L) q[L] = __float2int_rn(acc[L][v]);
  const long long hi = (long long)(q[0] * 128 + q[1]) * 16384 + (q[2] * 128 + q[3]);
  const long long lo = ((long long)(q[4] * 128 + q[5]) * 16384 + (q[6] * 128 + q[7])) * 128 + q[8];
  return oz_assemble_small(hi, lo, 35, E - 56);
}

// (double)f by integer operations (FP32 subnormals flush to zero)
__device__ __forceinline__ double oz_f2d(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xffu;
  if (e == 0) return __hiloint2double((int)(u & 0x80000000u), 0);
  return __hiloint2double((int)((u & 0x80000000u) | ((e + 896u) << 20) | ((u >> 3) & 0xfffffu)), (int)(u << 29));
}

// x or -x by the sign bit (no FP64 operation)
__device__ __forceinline__ double oz_neg_if(double x, bool neg) {
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)neg << 63));
}

}  // namespace jac
