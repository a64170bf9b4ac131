// pivot.cu -- one pivot block per CTA: the square factor and the inner one-sided Jacobi.
//
// For the pair (p, q) of a step, with X = [G_p G_q] (m x k) and A_P = X^* X (from the gram
// kernel):
//  1. convergence statistics of A_P: rotate the block iff some |a_ij| > tol sqrt(a_ii a_jj);
//  2. the Cholesky factor P^T A_P P = R^* R (Sec. 3.2), unpivoted (HF), with diagonal pivoting
//     over the whole block (HFC) or J_P-sign-pivoted (Algorithm 3.3, HFSC: diagonal pivoting
//     inside the J = +1 part, then inside the Schur complement of the J = -1 part, whose columns
//     are then taken in reverse order);
//  3. the pointwise one-sided Jacobi on the columns of R with respect to J_P (Sec. 2.1, the
//     "one-sided manner" of Sec. 2.2), trigonometric rotations (Eq. (2.1)) for equal signs and
//     hyperbolic ones otherwise, with the tanh = +-1 guard of Sec. 3.2, repeated until an inner
//     sweep rotates nothing (full block algorithm);
//  4. V_P = P W Pi (rows permuted back as Algorithm 3.4 states; Pi = the reversed order of the
//     J = -1 columns of Algorithm 3.3), J_P-unitary to FP64 accuracy when requested.
//
// GB300 placement.  Phases 1-3 (pivot_core) are a dependent chain of FP32 work: 4 KM threads, one
// block barrier per Cholesky step and per inner step.  Every FP32 pass runs on pairs of values
// (fma.rn.f32x2: two FMAs per issued instruction), since with at most one or two warps per
// scheduler the chain is bound by issue slots and latency, not by arithmetic.
//
// Precision of phases 2 and 3.  A_P is scaled, A_P = D (I + E) D with D = diag(fp32(sqrt(a_ii))),
// and only deviations from the identity enter the Cholesky step in FP32, so small off-diagonal
// entries keep their own relative precision.  The inner rotations act on the columns of R and of
// V as they stand; what a near-diagonal block needs beyond FP32 is carried beside the columns:
//   - the squared column norms as ||r_c||^2 = d_c^2 + cn_c, the deviation cn_c taken from the FP64
//     diagonal and moved by every rotation, so that the gap a_jj - a_ii of two nearly equal
//     columns keeps its relative precision;
//   - the diagonal of V - I, which the rounding of V_cc near 1 would lose, from the J-norm of the
//     column's other entries when the inner sweeps are done.
// The off-diagonal entries of R and V are FP32 numbers of their own size throughout.
//
// The transform that is applied to G in FP64 must be J-unitary in FP64 (phase 4, pivot_orth); it
// is corrected by Newton-Schulz,
//     V <- V - V J (V^T J V - J) / 2   (quadratic),
// on W = V - I: the residual M = W^T J + J W + W^T J W is formed in FP32 when max|W| <= 2^-20 and
// otherwise from FP16 digit products of W (oz_residual) or on the FP64 mma path (symmetric tiles
// only); the correction product itself is small and is formed in FP32.
#include "jacobi_common.cuh"
#include "pair_cache.cuh"
#include "ozaki.cuh"
#include "residual_sum.h"
#include "rotation.h"

namespace jac {

// ---- pairs of FP32 values in one 64-bit register ----------------------------------------------
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_make(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float f2_lo(f2 v) {
  return __uint_as_float((unsigned)v);
}
__device__ __forceinline__ float f2_hi(f2 v) {
  return __uint_as_float((unsigned)(v >> 32));
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// (float)x by integer operations (round to nearest, ties away from zero) for x of FP32 normal
// size or zero; `slow` is set for any other x (an FP64 conversion per entry costs ~0.6 clocks of
// the SM's FP64 pipe: 2.5k clocks for a 64 x 64 block)
__device__ __forceinline__ float d2f_fast(double x, bool& slow) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), m = hi & 0x7fffffffu;
  slow |= (m - (897u << 20)) >= (253u << 20) && (m | lo) != 0;
  const unsigned b = (((m - (896u << 20)) << 3) | (lo >> 29)) + ((lo >> 28) & 1u);
  return __uint_as_float(m < (897u << 20) ? 0u : (b | (hi & 0x80000000u)));
}

// ---- the core: statistics, Cholesky, inner Jacobi ---------------------------------------------
// Pivot capacity KM (largest k = w_p + w_q of the class): 4 KM threads; KM / 2 pair slots of LPP lanes
// each, R rows of both columns per lane, once for the columns of R (the first 2 KM threads) and once
// for those of V.
template <int KM>
struct PivotDim {
  static constexpr int LPP = 4;
  static constexpr int R = KM / LPP;
  static constexpr int H = R / 2;        // row pairs per lane
  static constexpr int P2 = KM / 2;      // pair slots
  static constexpr int NT = 4 * KM;      // threads
  static constexpr int NF = P2 * LPP;    // threads of the columns of R
  static constexpr int NW = NT / 32;
  static constexpr int LDT = KM + 4;     // Schur columns of the pivots (floats; 16-byte aligned)
  static constexpr int LDW = KM + 4;     // columns of W = V - I (floats; 16-byte aligned)
  static constexpr int TX = KM / 4;      // Cholesky tile of a thread: RU rows x 4 columns
  static constexpr int RU = KM / 16;
  static constexpr int MB = KM * P2;     // floats of one mailbox: a column of every slot
  static_assert(TX * 16 == NT && 2 * NF == NT && R % 4 == 0, "tile and lane layout");
};

// Block barrier of the inner sweep, where the two halves of the threads wait in code of their own.
template <int KM>
__device__ __forceinline__ void half_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(PivotDim<KM>::NT) : "memory");
}

// N floats (2 or 4) from shared memory
template <int N>
__device__ __forceinline__ void load_n(float (&v)[N], const float* p) {
  if constexpr (N == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  } else {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  }
}

template <int KM>
struct alignas(16) PivotState {
  using D = PivotDim<KM>;
  int4 mst[2][D::P2];   // traveling column of each slot: index, cn, d, sign
  float colb[2][KM];    // two-float factorization: pivot column of a step (double-buffered)
  float cold[2][KM];    // ... its low parts
  int4 piv[KM];         // Cholesky step i: pivot column, 1 / r, r (floats)
  float dd[KM];         // d_c
  float fid[KM];        // fp32(1 / d_c), 0 beyond k
  float ed[KM];         // e_cc
  float cn0[KM];        // a_cc - d_c^2
  double adiag[KM];
  int perm[KM];
  int lpos[KM];         // column at logical position l
  int linv[KM];         // logical position of column c
  int jphys[KM];        // signs in pivot order
  int jloc[KM];         // signs in local order
  int pres[D::P2];      // block-oriented cross step: columns of block p (pivot order) per slot
  int ptrav[D::P2];     // ... and of block q
  float4 prm[2][D::P2]; // rotation of each slot's pair: c, q12, q21 (double-buffered)
  int2 back[D::P2];     // places of a slot's columns at the start of an inner sweep
  float red_f[D::NW][4];
  int red_i[D::NW][2];
  double trs[2];
  int k, bad;
  long long t_core;     // clock at the end of the core
  PairStat st;          // kept by thread 0
};

template <int KM>
struct alignas(16) PivotWork {  // dead outside the core
  using D = PivotDim<KM>;
  union {
    float colh[KM * D::LDT];  // colh[i LDT + c]: Schur column of pivot i; times 1 / r, row i of R~
    float mb[2][2][D::MB];   // column mailboxes of the inner sweep: R, V (double-buffered)
  };
};

__device__ __forceinline__ float rsqrt_ftz(float x) {  // arguments of FP32 normal size
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// sum over the LPP lanes of a pair slot (aligned lane groups)
template <int LPP>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = LPP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---- two-float numbers (hi + lo, |lo| <= ulp(hi) / 2: about 48 bits) ---------------------------
__device__ __forceinline__ void ff_renorm(float& h, float& l) {
  const float s = h + l;
  l = l - (s - h);
  h = s;
}
__device__ __forceinline__ void ff_mul(float ah, float al, float bh, float bl, float& h, float& l) {
  h = ah * bh;
  l = fmaf(ah, bh, -h);
  l = fmaf(ah, bl, fmaf(al, bh, l));
  ff_renorm(h, l);
}
__device__ __forceinline__ void ff_sub(float& sh, float& sl, float ph, float pl) {  // s -= p
  const float d = sh - ph, bb = d - sh;
  const float e = (sh - (d - bb)) - (ph + bb);
  sh = d;
  sl = (sl + e) - pl;
  ff_renorm(sh, sl);
}
// 1 / sqrt(s): one Newton step on the FP32 seed, the residual formed in two floats
__device__ __forceinline__ void ff_rsqrt(float sh, float sl, float& h, float& l) {
  const float y = rsqrtf(sh);
  const float ph = y * y, pl = fmaf(y, y, -ph);
  const float qh = sh * ph, ql = fmaf(sh, ph, -qh);
  const float e = ((1.0f - qh) - ql) - fmaf(sh, pl, sl * ph);
  h = y;
  l = 0.5f * y * e;
  ff_renorm(h, l);
}

// The Cholesky factor of a block that FP32 cannot factor (a Schur pivot below 64 eps_32 of its
// diagonal entry), in two-float arithmetic: as the FP32 factorization of pivot_core (same tiles, same
// orders), on A_P scaled by powers of two.  Leaves row i of R~ in colh (FP32, R = R~ D with D =
// diag(dd), its 1 / r taken as 1) and the order in piv; sm.bad is set when a Schur pivot falls below 2^-36 of its diagonal
// entry (the FP64 pivot kernel then decides) and cleared otherwise.
// Square Gaussian factors of order 33..64 are often beyond FP32 in their first sweep (kappa(A~) above
// 2.6e5), and there the FP64 pivot took 1 to 3 ms per block (704 FP64 operations per pair of
// columns and step at ~1.6 per clock): 1000 problems of orders 8..128 spent 42% of their time in
// it.  This factorization costs ~60k clocks, and the FP32 rotations that follow bring the block
// within FP32's reach for the next sweep.
template <int KM>
__device__ __noinline__ void chol_two_float(PivotState<KM>& sm, float* colh, const double* A, int apld, int k, int npos,
                                            int factor) {
  using D = PivotDim<KM>;
  constexpr int NW = D::NW, TX = D::TX, RU = D::RU, LDT = D::LDT;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tx = tid % TX, ty = tid / TX, c0 = 4 * tx, r0 = RU * ty;
  const bool signpiv = (factor == 2), pivsel = factor != 0;
  // power-of-two scale near d_c: 2^-e_c
  auto pscale = [&](int c) { return __int_as_float(0x7f000000 - (__float_as_int(sm.dd[c]) & 0x7f800000)); };
  float H[RU][4], L[RU][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      const int i_ = r0 + u, j_ = c0 + j;
      const bool in = i_ < k && j_ < k;
      const double a = in ? __ldg(A + (size_t)j_ * apld + i_) : 0.0;
      const double b = a * (double)pscale(in ? i_ : 0) * (double)pscale(in ? j_ : 0);  // exact
      H[u][j] = (float)b;
      L[u][j] = (float)(b - (double)H[u][j]);
    }
  float dh[2], dl[2], dq[2], d0[2];
  bool al[2];
#pragma unroll
  for (int w = 0; w < KM / 32; ++w) {
    const int c = lane + 32 * w;
    const float ps = pscale(c < k ? c : 0);
    const double b = c < k ? sm.adiag[c] * (double)ps * (double)ps : 1.0;
    dh[w] = (float)b;
    dl[w] = (float)(b - (double)dh[w]);
    d0[w] = dh[w];
    dq[w] = 1.0f / (ps * ps);
    al[w] = c < k;
  }
  auto next_pivot = [&](int i) -> int {
    if (!pivsel) return i;
    unsigned key = 0;
#pragma unroll
    for (int w = 0; w < KM / 32; ++w) {
      const int c = lane + 32 * w;
      const bool in = al[w] && (!signpiv || ((i < npos) == (c < npos)));
      if (in) key = max(key, (__float_as_uint(fmaxf(dq[w] * dh[w], 0.0f)) & 0xFFFFFFC0u) | (unsigned)(63 - c));
    }
    return 63 - (int)(__reduce_max_sync(0xffffffffu, key) & 63u);
  };
  __syncthreads();  // the failed factorization's columns and rows are no longer read
  if (tid == 0) sm.bad = 0;
  int p = next_pivot(0);
  for (int i = 0; i < k; ++i) {
    const int b = i & 1;
    if (tx == (p >> 2)) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if ((p & 3) == j) {
#pragma unroll
          for (int u = 0; u < RU; ++u) {
            sm.colb[b][r0 + u] = H[u][j];
            sm.cold[b][r0 + u] = L[u][j];
          }
        }
    }
    // the smallest acceptable pivot, from the lane that carries column p
    const float dp = __shfl_sync(0xffffffffu, (KM == 64 && p >= 32) ? d0[KM / 32 - 1] : d0[0], p & 31);
    __syncthreads();
    const float ph = sm.colb[b][p], pl = sm.cold[b][p];
    if (!(ph > 1.4551915e-11f * dp)) {
      if (tid == 0) sm.bad = 1;
      break;  // uniform
    }
    float yh, yl;
    ff_rsqrt(ph, pl, yh, yl);
    float th[2], tl[2];
#pragma unroll
    for (int w = 0; w < KM / 32; ++w) {
      const int c = lane + 32 * w;
      ff_mul(sm.colb[b][c], sm.cold[b][c], yh, yl, th[w], tl[w]);
      float qh, ql;
      ff_mul(th[w], tl[w], th[w], tl[w], qh, ql);
      ff_sub(dh[w], dl[w], qh, ql);
      al[w] = al[w] && c != p;
    }
    const int pn = (i + 1 < k) ? next_pivot(i + 1) : 0;
    if (warp == i % NW) {
#pragma unroll
      for (int w = 0; w < KM / 32; ++w) {
        const int c = lane + 32 * w;
        // R column c is t 2^e_c; colh holds it relative to d_c
        const float t = c < k ? th[w] / (pscale(c) * sm.dd[c]) : 0.0f;
        colh[i * LDT + c] = t;
        if (c == p) sm.piv[i] = make_int4(p, __float_as_int(1.0f), __float_as_int(t), 0);
      }
    }
    float ch[4], cl[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) ff_mul(sm.colb[b][c0 + j], sm.cold[b][c0 + j], yh, yl, ch[j], cl[j]);
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      float rh, rl;
      ff_mul(sm.colb[b][r0 + u], sm.cold[b][r0 + u], yh, yl, rh, rl);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float q = rh * ch[j], e = fmaf(rh, cl[j], fmaf(rl, ch[j], fmaf(rh, ch[j], -q)));
        ff_sub(H[u][j], L[u][j], q, e);
      }
    }
    p = pn;
  }
  __syncthreads();
}

// Phases 1-3 of one pair, run by all 4 KM threads of a CTA.  Returns (uniformly) 0 when V_P was
// formed: W = V - I in Wf (column c at c LDW, pivot order), the orders in sm; 2 when the block was
// handed over to the FP64 pivot kernel; 1 otherwise (no rotation, or a reported error).  A32: A_P is
// read from shared memory (FP32, column c at c LDW), else from the Gram kernel's output.  `skip` and
// the statistics of the pair are written here unless the result is 0.
template <int KM, bool A32>
__device__ __forceinline__ int pivot_core(PivotState<KM>& sm, PivotWork<KM>& wk, const float* As, float* Wf,
                                          const JacProb& a, int s, int pair, const PivotParams& pp) {
  using D = PivotDim<KM>;
  constexpr int NW = D::NW, TX = D::TX, RU = D::RU, LDT = D::LDT, LDW = D::LDW, P2 = D::P2;
  constexpr int LPP = D::LPP, R = D::R, H = D::H;
  unsigned* err = a.pflags;
  PairStat* stats = a.stats + (size_t)s * a.half;
  const long long t_start = clock64();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tx = tid % TX, ty = tid / TX, c0 = 4 * tx, r0 = RU * ty;

  // ---- 1. load A_P, scaled matrix E, statistics ----------------------------------------------
  // The addresses depend on the pair slot only: these loads (the whole tile, entries beyond k
  // unused) are issued before the dependent lookups of the pair's blocks
  const double* A = a.Ap + (size_t)pair * a.apld * a.apld;
  float e[RU][4];
  double adg = 1.0;
  bool slow = false;
  double2 av[4][RU / 2];
  if constexpr (!A32) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < RU / 2; ++u)
        av[j][u] = __ldg(reinterpret_cast<const double2*>(A + (size_t)(c0 + j) * a.apld + r0 + 2 * u));
    if (tid < KM) adg = __ldg(A + (size_t)tid * a.apld + tid);
  }
  const int* sp = a.pairs + (size_t)s * a.half * 2;
  const int p_ = sp[2 * pair], q_ = sp[2 * pair + 1];
  const int op = a.boff[p_], wp = a.boff[p_ + 1] - op, oq = a.boff[q_], wq = a.boff[q_ + 1] - oq;
  const int k = wp + wq;
  if (k > KM) {  // the driver assigns classes by k; reported, never trapped
    if (tid == 0) {
      atomicOr(err, JAC_DEVERR_INNER_LIMIT);
      a.skip[pair] = 1;
    }
    return 1;
  }
  if (tid == 0) {
    sm.bad = 0;
    sm.k = k;
  }
  if (tid < P2) {
    sm.pres[tid] = -1;
    sm.ptrav[tid] = -1;
  }
  __syncthreads();  // bad cleared
  if constexpr (!A32) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        bool sl = false;
        const float x = d2f_fast((u & 1) ? av[j][u / 2].y : av[j][u / 2].x, sl);
        const bool in = r0 + u < k && c0 + j < k;
        e[u][j] = in ? x : 0.0f;
        slow |= in && sl;
      }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v[RU];
      load_n<RU>(v, As + (c0 + j) * LDW + r0);
#pragma unroll
      for (int u = 0; u < RU; ++u) e[u][j] = v[u];
    }
    if (tid < k) adg = (double)As[tid * LDW + tid];
  }
  double tr = 0.0;
  if (tid < KM) {
    float d = 1.0f, fid = 0.0f, ed = 0.0f, cn = 0.0f;
    int j = 1;
    if (tid < k) {
      j = a.Js[tid < wp ? op + tid : oq + (tid - wp)];
      if (!(adg > 0.0) || !(adg < 1.0e300)) atomicOr(&sm.bad, 1);
      d = sqrtf((float)adg);
      fid = 1.0f / d;
      // a_ii - d_i^2 is exact in FP64 (both agree to FP32 accuracy), rounded once
      const double d2 = (double)d * (double)d;
      cn = (float)(adg - d2);
      ed = cn / (float)d2;
      tr = adg;
    }
    sm.dd[tid] = d;
    sm.fid[tid] = fid;
    sm.ed[tid] = ed;
    sm.cn0[tid] = cn;
    sm.adiag[tid] = adg;
    sm.jloc[tid] = j;
  }
  __syncthreads();
  if (sm.bad) {
    if (tid == 0) {
      atomicOr(err, JAC_DEVERR_NOTPD);
      a.skip[pair] = 1;
      PairStat st = {};
      st.evaluated = 1;
      stats[pair] = st;
    }
    return 1;
  }
  if constexpr (!A32) {
    if (slow) {  // some entry outside the FP32 normal range
#pragma unroll 1
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int u = 0; u < RU; ++u) {
          const float x = (r0 + u < k && c0 + j < k) ? (float)__ldg(A + (size_t)(c0 + j) * a.apld + r0 + u) : 0.0f;
          if (j == 0) e[u][0] = x;
          else if (j == 1) e[u][1] = x;
          else if (j == 2) e[u][2] = x;
          else e[u][3] = x;
        }
    }
  }
  // off-diagonal e_ij = a_ij / (d_i d_j) in FP32: it is the scaled off-diagonal entry
  // |a_ij| / sqrt(a_ii a_jj) to FP32 accuracy, so it drives the statistics; only entries within
  // 2^-12 of the threshold are re-decided in FP64.  Both triangles are counted (sums halved).
  const double tol = pp.tol > 0.0 ? pp.tol : fmax((double)a.n, pp.tol_m * sqrt((double)a.mp)) * pp.tol_eps;
  const float tolf = (float)tol;
  float mx = 0.0f, oc = 0.0f, od = 0.0f;
  bool hit = false;
  unsigned near = 0;
  {
    float fr[RU];
    load_n<RU>(fr, &sm.fid[r0]);
    const float4 fc4 = *reinterpret_cast<const float4*>(&sm.fid[c0]);
    const float fc[4] = {fc4.x, fc4.y, fc4.z, fc4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const int i_ = r0 + u, j_ = c0 + j;
        const float x = (i_ < k && j_ < k && i_ != j_) ? e[u][j] : 0.0f;
        const float x2 = x * x, v = x * fr[u] * fc[j], r = fabsf(v);
        e[u][j] = v;
        mx = fmaxf(mx, r);
        hit |= r > tolf;
        near |= (fabsf(r - tolf) <= tolf * 2.44140625e-4f) ? 1u << (RU * j + u) : 0u;
        if ((i_ < wp) != (j_ < wp)) oc += x2;
        else od += x2;
      }
    if (near) {
      hit = false;
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int u = 0; u < RU; ++u)
          if (!((near >> (RU * j + u)) & 1u)) hit |= fabsf(e[u][j]) > tolf;
      for (unsigned m = near; m; m &= m - 1) {
        const int b = __ffs((int)m) - 1, i_ = r0 + b % RU, j_ = c0 + b / RU;
        const double ad = A32 ? (double)As[j_ * LDW + i_] : __ldg(A + (size_t)j_ * a.apld + i_);
        hit |= ad * ad > tol * tol * sm.adiag[i_] * sm.adiag[j_];
      }
    }
  }
  // npos: the J = +1 columns come first
  int npos = __popc(__ballot_sync(0xffffffffu, lane < k && sm.jloc[lane] > 0));
  if constexpr (KM == 64) npos += __popc(__ballot_sync(0xffffffffu, lane + 32 < k && sm.jloc[lane + 32] > 0));
  mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
  hit = __any_sync(0xffffffffu, hit);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    oc += __shfl_xor_sync(0xffffffffu, oc, o);
    od += __shfl_xor_sync(0xffffffffu, od, o);
  }
  if (warp < KM / 32) tr = warp_sum_d(tr);
  if (lane == 0) {
    sm.red_f[warp][0] = mx;
    sm.red_f[warp][1] = oc;
    sm.red_f[warp][2] = od;
    sm.red_i[warp][0] = hit;
    if (warp < KM / 32) sm.trs[warp] = tr;
  }
  __syncthreads();
  mx = oc = od = 0.0f;
  hit = false;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    mx = fmaxf(mx, sm.red_f[w][0]);
    oc += sm.red_f[w][1];
    od += sm.red_f[w][2];
    hit |= sm.red_i[w][0] != 0;
  }
  const long long t_stats = clock64();
  if (tid == 0) {
    PairStat& st = sm.st;
    st.max_scaled = (double)mx;
    st.off2_cross = 0.5 * (double)oc;
    st.off2_diag = 0.5 * (double)od;
    st.trace = sm.trs[0] + (KM == 64 ? sm.trs[1] : 0.0);
    st.rotations = 0;
    st.inner_sweeps = 0;
    st.ns_steps = 0;
    st.active = hit ? 1 : 0;
    st.evaluated = 1;
    st.cyc[0] = t_stats - t_start;
    st.cyc[1] = st.cyc[2] = st.cyc[3] = 0;
    if (!hit) {
      a.skip[pair] = 1;
      pair_record(a, s, pair, false);
      stats[pair] = st;
    }
  }
  if (!hit) return 1;

  // ---- 2. scaled, optionally sign-pivoted Cholesky in FP32 -----------------------------------
  // Right-looking on unpermuted storage, the whole symmetric matrix E (both triangles) in
  // registers: thread (ty, tx) holds rows r0.. and columns c0.. .  Step i with pivot column p: the
  // threads of column p have published it (as row i of colh, one barrier per step), every thread
  // scales it to t = s_p / sqrt(s_pp), and t_r t_c comes off its tile.  Every warp carries the shifted
  // Schur diagonal s_cc of all columns (lane: c = lane, lane + 32) with the same operations, so the
  // pivot search of the next step needs no barrier: a warp max-reduction of keys, the value's bits
  // above the low 6 (order-preserving for v >= 0, negative for v < 0) and 63 - c, the largest unscaled
  // Schur diagonal d_c^2 (1 + s_cc) in the sign group of the step (sign pivoting, Algorithm 3.3) or
  // among all remaining columns (diagonal pivoting, HFC), ties to the smaller index.
  // A step is one chain: barrier, column, rsqrt, key, search, publish.  What is not on it stays out
  // of its way: the next column is published with its own update first and the tile's update
  // follows after the loads of the next step, the rows of R~ need no stores of their own, no branch
  // but the loop's.  ~410 clocks per step; left-looking with the rows in shared memory it took 940.
  const bool signpiv = (pp.factor == 2), diagpiv = (pp.factor == 1), pivsel = signpiv || diagpiv;
  // the tile of E: its shifted diagonal into e
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int u = 0; u < RU; ++u)
      if (r0 + u == c0 + j) e[u][j] = sm.ed[c0 + j];
  float dv0 = sm.ed[lane], dq0 = sm.dd[lane] * sm.dd[lane], dv1 = 0.0f, dq1 = 0.0f;
  bool al0 = lane < k, al1 = false;
  if constexpr (KM == 64) {
    dv1 = sm.ed[lane + 32];
    dq1 = sm.dd[lane + 32] * sm.dd[lane + 32];
    al1 = lane + 32 < k;
  }
  auto next_pivot = [&](int i) -> int {
    if (!pivsel) return i;
    const bool first = i < npos;
    auto key_of = [&](bool alive, float dq, float dv, int c) {
      const bool in = alive && (!signpiv || first == (c < npos));
      return in ? (int)((__float_as_uint(fmaf(dq, dv, dq)) & 0xFFFFFFC0u) | (unsigned)(63 - c)) : (int)0x80000000;
    };
    int key = key_of(al0, dq0, dv0, lane);
    if constexpr (KM == 64) key = max(key, key_of(al1, dq1, dv1, lane + 32));
    return 63 - (__reduce_max_sync(0xffffffffu, key) & 63);  // signed: a negative value never wins
  };
  auto pick = [](int p, const float(&x)[4]) {  // x[p & 3] by selects: a jump on it costs ~50 clocks
    const float lo = (p & 1) ? x[1] : x[0], hi = (p & 1) ? x[3] : x[2];
    return (p & 2) ? hi : lo;
  };
  auto publish = [&](int i, int p, const float(&x)[RU]) {
    if (tx == (p >> 2)) {
      if constexpr (RU == 4) *reinterpret_cast<float4*>(&wk.colh[i * LDT + r0]) = make_float4(x[0], x[1], x[2], x[3]);
      else *reinterpret_cast<float2*>(&wk.colh[i * LDT + r0]) = make_float2(x[0], x[1]);
    }
  };
  int p = next_pivot(0);
  float tu[RU], tc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  bool bad = false;
  {
    float x[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      x[u] = pick(p, e[u]);
      tu[u] = 0.0f;
    }
    publish(0, p, x);
  }
  for (int i = 0; i < k; ++i) {
    __syncthreads();
    const float* col = wk.colh + i * LDT;
    const float spp = col[p], v0 = col[lane], v1 = (KM == 64) ? col[lane + (KM - 32)] : 0.0f;
    float vc[4], vr[RU];
    load_n<4>(vc, &col[c0]);
    load_n<RU>(vr, &col[r0]);
#pragma unroll
    for (int j = 0; j < 4; ++j)  // the previous step's update of the tile
#pragma unroll
      for (int u = 0; u < RU; ++u) e[u][j] = fmaf(tu[u], tc[j], e[u][j]);
    // The scaled Schur pivot is 1 / (A~^-1)_pp >= 1 / kappa(A~).  Below 64 eps_32 the column is
    // in the span of the previous ones at the precision of this factorization: a more precise one
    // takes the block (below).
    const float piv1 = 1.0f + spp;
    bad |= !(piv1 > 3.8146973e-6f);
    const float rinv = rsqrt_ftz(fmaxf(piv1, 3.8146973e-6f));  // 1 / r
    const float t0 = v0 * rinv, t1 = v1 * rinv;
    dv0 = fmaf(-t0, t0, dv0);
    dv1 = fmaf(-t1, t1, dv1);
    al0 = al0 && lane != p;
    al1 = al1 && lane + 32 != p;
    if (tid == 0) sm.piv[i] = make_int4(p, __float_as_int(rinv), __float_as_int(piv1 * rinv), 0);
    const int pn = next_pivot(i + 1) & (KM - 1);
#pragma unroll
    for (int j = 0; j < 4; ++j) tc[j] = -vc[j] * rinv;
#pragma unroll
    for (int u = 0; u < RU; ++u) tu[u] = vr[u] * rinv;
    p = pn;
    const float tp = pick(p, tc);
    float x[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) x[u] = fmaf(tu[u], tp, pick(p, e[u]));
    if (i + 1 < k) publish(i + 1, p, x);
  }
  if (tid == 0) sm.bad = bad ? 1 : 0;  // the same in every thread
  __syncthreads();
  if constexpr (!A32) {
    if (sm.bad && pp.ns_mode) chol_two_float<KM>(sm, wk.colh, A, a.apld, k, npos, pp.factor);
  }
  if (sm.bad) {  // handed over to the FP64 pivot kernel, which decides on rank deficiency
    if (tid == 0) {
      a.skip[pair] = 2;
      atomicOr(err, JAC_DEVERR_HANDOVER);
      sm.st.cyc[1] = clock64() - t_stats;
      stats[pair] = sm.st;
    }
    return 2;
  }
  // Orders.  Block-oriented steps after the first of a sweep rotate only the cross pairs (one
  // column of block p, one of block q): block p's columns become the residents of the ring, block
  // q's the travelers, each in pivot order.  Diagonal pivoting mixes the signs: the output order
  // puts the pivot-order columns back on positions of their own sign (positives, then negatives,
  // each in pivot order), so that V_P^* J_P V_P = J_P in the block's local order (the reordering of
  // HFC).  Sign pivoting takes the J = -1 columns in reverse.
  const bool cross_only = pp.oriented && s > 0;
  if (tid < k) sm.perm[tid] = sm.piv[tid].x;
  __syncthreads();
  {
    auto mask64 = [&](auto f) -> unsigned long long {  // f(position) over the k positions
      unsigned long long m = __ballot_sync(0xffffffffu, lane < k && f(lane < k ? lane : 0));
      if constexpr (KM == 64)
        m |= (unsigned long long)__ballot_sync(0xffffffffu, lane + 32 < k && f(lane + 32 < k ? lane + 32 : 0)) << 32;
      return m;
    };
    const unsigned long long mpos = mask64([&](int c) { return sm.jloc[sm.perm[c]] > 0; });
    const unsigned long long mp = mask64([&](int c) { return sm.perm[c] < wp; });
    if (tid < k) {
      const unsigned long long below = (1ull << tid) - 1;
      const bool pos = (mpos >> tid) & 1;
      int l = tid;
      if (diagpiv) l = pos ? __popcll(mpos & below) : npos + __popcll(~mpos & below);
      else if (signpiv && tid >= npos) l = k - 1 - (tid - npos);
      sm.lpos[l] = tid;
      sm.linv[tid] = l;
      sm.jphys[tid] = pos ? 1 : -1;
      if (cross_only) {
        if ((mp >> tid) & 1) sm.pres[__popcll(mp & below)] = tid;
        else sm.ptrav[__popcll(~mp & below)] = tid;
      }
    } else if (tid < KM) {
      sm.jphys[tid] = 1;
    }
  }
  __syncthreads();
  const long long t_chol = clock64();

  // ---- 3. inner one-sided Jacobi (FP32) -------------------------------------------------------
  // inner threshold: at most half the outer one (so that a pair flagged in FP64 is rotated in
  // FP32), at least the FP32 noise level of the dot products
  const float tol_in = fmaxf(0.5f * tolf, 64.0f * 5.9604645e-8f * mx);
  // The columns live in registers: pair slot q (LPP lanes of a warp) holds a resident and a
  // traveler column of R and of V, R rows per lane (row l R + u in lane l), as row pairs.  An inner
  // sweep is a recursive cross ordering of the k columns over p = ceil(k / 2) slots: the travelers of a
  // group of g slots (g = p at first) go round its ring, so every resident meets every traveler of
  // the group in g steps; then each group splits in two of ceil(g / 2) slots, its residents pairing
  // among themselves in the first and its travelers in the second.  Every pair meets once in
  // p + ceil(p / 2) + ... + 1 steps, and between steps each slot passes at most one column to one
  // other slot through a shared-memory mailbox: one barrier per step.  A group of g slots lies in a
  // range of w >= g, w = p2, p2/2, ..., 1 (p2: the power of two >= p): its i-th slot is i if p is p2, and
  // else i with its bits reversed.  Then slots of odd i lie w/2 above those of even i, so the split
  // sends columns w/2 slots up or down for every g, and what the odd ones hold stays among the
  // first ceil(g / 2).  An empty place holds a zero column that rests.  The logical order of Algorithm
  // 3.3 (reversed J = -1 part) gives the initial placement: position i is the resident of slot i
  // (i < p) or the traveler of slot i - p.  If p < p2 the columns end a sweep spread over p2 slots
  // and go back to where they began before the next.
  // Orders 33..64 take 50 steps per sweep on average, where a ring of p2 slots takes 63: 4000 problems
  // of orders 8..128 in FP32 31.4 ms, now 27.0, in FP64 74.1 ms, now 68.5.
  // What bounds a step is its chain: mailbox, dot product and its reduction, the parameters, the
  // rotation, mailbox, barrier.  The columns of V are not on it: they belong to the second half of
  // the threads, which rotate them one barrier later, with the parameters the first half left in
  // shared memory, in the shadow of the first half's next step.  ~700 clocks per step for a 64-column
  // block; rotating both in the same threads, with the parameters by way of the tangent, took 965 (and
  // spreading the columns over 32 lanes, to keep the ring in registers, 1235: five shuffle rounds
  // and the exchange of the parameters cost more than the mailboxes).
  const bool is_f = tid < D::NF;
  const int slot = (is_f ? tid : tid - D::NF) / LPP, l = tid % LPP;
  const int np = (k + 1) / 2, p2 = 1 << (32 - __clz(np - 1));
  // the i-th slot of a range of w slots, and the i of a slot
  auto order = [&](int i, int w) { return np == p2 ? i : (int)((__brev((unsigned)i) >> __clz(w)) >> 1); };
  auto start_i = [&]() {
    const int i = order(slot, p2);
    return (slot >= p2 || i >= np) ? -1 : cross_only ? sm.pres[i] : sm.lpos[i];
  };
  auto start_j = [&]() {
    const int i = order(slot, p2);
    return (slot >= p2 || i >= np) ? -1 : cross_only ? sm.ptrav[i] : (i + np < k ? sm.lpos[i + np] : -1);
  };
  // where the traveler of this slot goes in the ring of its group, five bits per level (the reversal
  // of bits at the start of each level cost its chain ~90 clocks)
  unsigned rings = 0;
  for (int w = p2, g = np, sh = 0; w >= 1; w >>= 1, g = (g + 1) >> 1, sh += 5) {
    const int i = order(slot & (w - 1), w);
    const int nxt = i < g ? (slot & ~(w - 1)) + order(i + 1 == g ? 0 : i + 1, w) : slot;
    rings |= (unsigned)nxt << sh;
  }
  // block-oriented: one inner sweep; after the first step of an outer sweep only the ring of
  // its first level (every column of block p meets every column of block q once)
  const int w_last = cross_only ? p2 : 1;
  const int max_inner = pp.oriented ? 1 : JAC_INNER_MAX_SWEEPS;
  f2 xi[H], xj[H];  // resident and traveler of this half's columns
  float cni = 0.0f, cnj = 0.0f, si = 1.0f, sj = 1.0f;  // ||r||^2 = s^2 + cn
  int ci = start_i(), cj = start_j(), ji = 1, jj = 1;
  if (is_f) {
    auto load_col = [&](int c, f2(&f)[H], float& cn, float& d, int& sg) {
      const int pc = c >= 0 ? sm.perm[c] : 0;
      cn = c >= 0 ? sm.cn0[pc] : 0.0f;
      d = c >= 0 ? sm.dd[pc] : 1.0f;
      sg = c >= 0 ? sm.jphys[c] : 1;
#pragma unroll
      for (int u = 0; u < H; ++u) {
        float r[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {  // R[row][c] = R~[row][c] d_c, upper triangular in pivot order
          const int row = l * R + 2 * u + t;
          const int4 pv = sm.piv[row];
          const float v = (row == c) ? __int_as_float(pv.z) : wk.colh[row * LDT + pc] * __int_as_float(pv.y);
          r[t] = (row <= c) ? v * d : 0.0f;
        }
        f[u] = f2_make(r[0], r[1]);
      }
    };
    load_col(ci, xi, cni, si, ji);
    load_col(cj, xj, cnj, sj, jj);
  } else {
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const int row = l * R + 2 * u;
      xi[u] = f2_make(row == ci ? 1.0f : 0.0f, row + 1 == ci ? 1.0f : 0.0f);
      xj[u] = f2_make(row == cj ? 1.0f : 0.0f, row + 1 == cj ? 1.0f : 0.0f);
    }
  }
  __syncthreads();  // the Cholesky rows are read; the mailboxes take their place
  int total_rot = 0, inner = 0, buf = 0;
  // a column's mailbox: 16-byte chunk q of lane l at ((q P2 + slot) LPP + l): a quarter warp writes
  // and reads 128 consecutive bytes
  auto box = [&](int b, int q, int sl) {
    return reinterpret_cast<ulonglong2*>(wk.mb[b][is_f ? 0 : 1]) + ((q * P2 + sl) * LPP + l);
  };
  auto put = [&](int b, int dst, const f2(&f)[H]) {
#pragma unroll
    for (int u = 0; u < H; u += 2) *box(b, u / 2, dst) = make_ulonglong2(f[u], f[u + 1]);
  };
  auto get = [&](int b, f2(&f)[H]) {
#pragma unroll
    for (int u = 0; u < H; u += 2) {
      const ulonglong2 x = *box(b, u / 2, slot);
      f[u] = x.x;
      f[u + 1] = x.y;
    }
  };
  auto rotate = [&](float c, float s12, float s21) {
    const f2 q11 = f2_make(c, c), q12 = f2_make(s12, s12), q21 = f2_make(s21, s21);
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const f2 a_i = xi[u], a_j = xj[u];
      xi[u] = f2_fma(q11, a_i, f2_mul(q21, a_j));
      xj[u] = f2_fma(q11, a_j, f2_mul(q12, a_i));
    }
  };
  for (inner = 0; inner < max_inner; ++inner) {
    int my_rot = 0;       // per slot (uniform over its lanes)
    float my_max = 0.0f;  // largest scaled |a_ij| rotated
    if (is_f) {
      if (inner > 0) {
        // a norm that has moved far from its reference d^2 (nearly dependent columns) is no longer
        // resolved by d^2 + cn: take it from the column, with a new reference
        auto fresh = [&](const f2(&f)[H], float& cn, float& d) {
          f2 q0 = f2_mul(f[0], f[0]), q1 = f2_mul(f[1], f[1]);
#pragma unroll
          for (int u = 2; u < H; u += 2) {
            q0 = f2_fma(f[u], f[u], q0);
            q1 = f2_fma(f[u + 1], f[u + 1], q1);
          }
          const float q = group_sum<LPP>((f2_lo(q0) + f2_lo(q1)) + (f2_hi(q0) + f2_hi(q1)));
          if (!(fabsf(cn) < 0.75f * d * d) && q > 0.0f) {
            d = sqrtf(q);
            cn = fmaf(-d, d, q);
          }
        };
        fresh(xi, cni, si);
        fresh(xj, cnj, sj);
      }
      unsigned ring = rings;
      for (int w = p2, g = np; w >= w_last; w >>= 1, g = (g + 1) >> 1, ring >>= 5) {
        const int nxt = ring & 31;
        for (int st_ = 0; st_ < g; ++st_) {
          // ---- rotate the pair (ci, cj) of this slot; what does not depend on the dot product first.
          // One branch-free path for both kinds (rotation.h): the slots of a warp never split on the
          // sign pattern.
          const bool trig = ji == jj;
          const float sg = trig ? 1.0f : -1.0f, sg4 = 4.0f * sg;
          const float aii = fmaf(si, si, cni), ajj = fmaf(sj, sj, cnj);
          const float x = trig ? (sj - si) * (sj + si) + (cnj - cni) : aii + ajj;
          const RotUnit ru = rot_unit(aii, ajj, x);
          // sign of the tangent: that of x (trigonometric), negative (hyperbolic)
          const unsigned tsign = trig ? __float_as_uint(x) & 0x80000000u : 0x80000000u;
          f2 d0 = f2_mul(xi[0], xj[0]), d1 = f2_mul(xi[1], xj[1]);
#pragma unroll
          for (int u = 2; u < H; u += 2) {
            d0 = f2_fma(xi[u], xj[u], d0);
            d1 = f2_fma(xi[u + 1], xj[u + 1], d1);
          }
          const float aij = group_sum<LPP>((f2_lo(d0) + f2_lo(d1)) + (f2_hi(d0) + f2_hi(d1)));
          const float scaled = fabsf(aij) * ru.rs;
          const bool rot = (ci | cj) >= 0 && scaled > tol_in;
          const RotAngle ra = rot_angle(ru, sg, sg4, fabsf(aij));
          const float c = rot ? ra.c : 1.0f;
          const float es = rot ? __uint_as_float(__float_as_uint(ra.s) ^ ((__float_as_uint(aij) & 0x80000000u) ^ tsign)) : 0.0f;
          const float q21 = -sg * es;
          if (l == 0) sm.prm[buf][slot] = make_float4(c, es, q21, 0.0f);
          rotate(c, es, q21);
          my_rot += rot ? 1 : 0;
          my_max = fmaxf(my_max, rot ? scaled : 0.0f);
          // a_ii' = a_ii - t |a_ij|, a_jj' = a_jj + t |a_ij| (trigonometric); both move by
          // t |a_ij| (hyperbolic: the J-trace is invariant); t = s / c.  Where the
          // guard acted a_ij is not annihilated: both norms are put out of range, so that the columns
          // rest until the next inner sweep takes them afresh
          const float ta = rot ? __uint_as_float(__float_as_uint(ra.s * ra.cinv * fabsf(aij)) ^ tsign) : 0.0f;
          const bool far = rot && ra.guard;
          cni = far ? 1.0e8f * si * si : fmaf(-sg, ta, cni);
          cnj = far ? 1.0e8f * sj * sj : cnj + ta;
          // ---- pass one column on: the traveler round the ring, or at the end of the group's
          // ring its split (first half: traveler to slot + w/2, which sends back its resident).  The
          // two cases are uniform over the block and keep code of their own: with one code for both,
          // the choice of the column split every warp
          if (st_ < g - 1) {
            put(buf, nxt, xj);
            if (l == 0) sm.mst[buf][nxt] = make_int4(cj, __float_as_int(cnj), __float_as_int(sj), jj);
            half_sync<KM>();
            const int4 m = sm.mst[buf][slot];
            get(buf, xj);
            cj = m.x;
            cnj = __int_as_float(m.y);
            sj = __int_as_float(m.z);
            jj = m.w;
          } else if (w > w_last) {
            const bool res = (slot & (w >> 1)) != 0;
            const int dst = slot ^ (w >> 1);
            if (res) put(buf, dst, xi);
            else put(buf, dst, xj);
            if (l == 0)
              sm.mst[buf][dst] = res ? make_int4(ci, __float_as_int(cni), __float_as_int(si), ji)
                                     : make_int4(cj, __float_as_int(cnj), __float_as_int(sj), jj);
            half_sync<KM>();
            const int4 m = sm.mst[buf][slot];
            if (res) {
              get(buf, xi);
              ci = m.x;
              cni = __int_as_float(m.y);
              si = __int_as_float(m.z);
              ji = m.w;
            } else {
              get(buf, xj);
              cj = m.x;
              cnj = __int_as_float(m.y);
              sj = __int_as_float(m.z);
              jj = m.w;
            }
          } else {
            half_sync<KM>();
          }
          buf ^= 1;
        }
      }
    } else {
      unsigned ring = rings;
      for (int w = p2, g = np; w >= w_last; w >>= 1, g = (g + 1) >> 1, ring >>= 5) {
        const int nxt = ring & 31;
        for (int st_ = 0; st_ < g; ++st_) {
          half_sync<KM>();  // the parameters of this step, the columns passed on in the previous one
          const float4 q = sm.prm[buf][slot];
          if (st_ > 0) {
            get(buf ^ 1, xj);
          } else if (w < p2) {  // the split that ended the ring of the range of 2 w slots
            if (slot & w) get(buf ^ 1, xi);
            else get(buf ^ 1, xj);
          }
          rotate(q.x, q.y, q.z);
          if (st_ < g - 1) {
            put(buf, nxt, xj);
          } else if (w > w_last) {
            if (slot & (w >> 1)) put(buf, slot ^ (w >> 1), xi);
            else put(buf, slot ^ (w >> 1), xj);
          }
          buf ^= 1;
        }
      }
    }
    // sweep totals: one count per slot (its lane 0)
    const int cnt = (int)__reduce_add_sync(0xffffffffu, (l == 0) ? (unsigned)my_rot : 0u);
    my_max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(my_max)));
    if (lane == 0) {
      sm.red_i[warp][1] = cnt;
      sm.red_f[warp][3] = my_max;
    }
    __syncthreads();
    int tot = 0;
    float dmax = 0.0f;
#pragma unroll
    for (int w = 0; w < NW / 2; ++w) {
      tot += sm.red_i[w][1];
      dmax = fmaxf(dmax, sm.red_f[w][3]);
    }
    __syncthreads();
    total_rot += tot;
    // done when nothing was rotated, or when every rotated pair was already so small that the
    // next sweep (quadratic convergence: off-diagonals ~ k delta^2) would find nothing above tol_in
    if (tot == 0 || (float)k * dmax * dmax <= tol_in) break;
    if (np < p2 && inner + 1 < max_inner) {  // back to the initial placement
      auto place = [&](int c) {  // slot, + KM for the traveler's place
        if (c < 0) return -1;
        const int q = sm.linv[c];
        return q < np ? order(q, p2) : order(q - np, p2) + KM;
      };
      if (is_f && l == 0) {
        const int di = place(ci), dj = place(cj);
        sm.back[slot] = make_int2(di, dj);
        if (di >= 0) sm.mst[di / KM][di % KM] = make_int4(ci, __float_as_int(cni), __float_as_int(si), ji);
        if (dj >= 0) sm.mst[dj / KM][dj % KM] = make_int4(cj, __float_as_int(cnj), __float_as_int(sj), jj);
      }
      __syncthreads();
      const int2 d = sm.back[slot];
      if (d.x >= 0) put(d.x / KM, d.x % KM, xi);
      if (d.y >= 0) put(d.y / KM, d.y % KM, xj);
      __syncthreads();
      const bool hi = start_i() >= 0, hj = start_j() >= 0;
#pragma unroll
      for (int u = 0; u < H; ++u) xi[u] = xj[u] = f2_make(0.0f, 0.0f);
      ci = cj = -1;
      cni = cnj = 0.0f;
      si = sj = 1.0f;
      ji = jj = 1;
      if (hi) {
        get(0, xi);
        const int4 m = sm.mst[0][slot];
        ci = m.x;
        cni = __int_as_float(m.y);
        si = __int_as_float(m.z);
        ji = m.w;
      }
      if (hj) {
        get(1, xj);
        const int4 m = sm.mst[1][slot];
        cj = m.x;
        cnj = __int_as_float(m.y);
        sj = __int_as_float(m.z);
        jj = m.w;
      }
      __syncthreads();
    }
  }
  if (!pp.oriented && inner >= JAC_INNER_MAX_SWEEPS && tid == 0) atomicOr(err, JAC_DEVERR_INNER_LIMIT);
  // which columns the slots of V hold now
  if (is_f && l == 0) sm.mst[0][slot] = make_int4(ci, cj, ji, jj);
  __syncthreads();
  // W = V - I.  The diagonal from the J-norm of the column, J_c sum_r J_r v_rc^2 = 1:
  // v_cc - 1 = -S / (1 + sqrt(1 - S)), S = J_c sum_{r != c} J_r v_rc^2, where S is small; the
  // rounded v_cc itself would lose W_cc ~ S / 2 below 2^-24
  auto finish = [&](int c, int sg, const f2(&w)[H]) {
    float S1 = 0.0f;
    float v[R];
#pragma unroll
    for (int u = 0; u < H; ++u) {
      v[2 * u] = f2_lo(w[u]);
      v[2 * u + 1] = f2_hi(w[u]);
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int row = l * R + u;
      const float q = (row == c) ? 0.0f : v[u] * v[u];
      S1 += (sm.jphys[row] < 0) ? -q : q;
    }
    S1 = group_sum<LPP>(S1) * (float)sg;
    const float wd = -__fdividef(S1, 1.0f + sqrtf(1.0f - fminf(S1, 0.5f)));
    if (c < 0) return;
#pragma unroll
    for (int u = 0; u < R; ++u) {
      if (l * R + u == c) v[u] = (v[u] > 0.0f && fabsf(S1) < 0.5f) ? wd : v[u] - 1.0f;
    }
#pragma unroll
    for (int u = 0; u < R; u += 4)
      *reinterpret_cast<float4*>(&Wf[c * LDW + l * R + u]) = make_float4(v[u], v[u + 1], v[u + 2], v[u + 3]);
  };
  if (!is_f) {
    const int4 m = sm.mst[0][slot];
    finish(m.x, m.z, xi);
    finish(m.y, m.w, xj);
  }
  const long long t_inner = clock64();
  if (tid == 0) {
    sm.st.rotations = total_rot;
    sm.st.inner_sweeps = (inner < max_inner) ? inner + 1 : max_inner;
    sm.st.cyc[1] = t_chol - t_stats;
    sm.st.cyc[2] = t_inner - t_chol;
    sm.t_core = t_inner;
  }
  return 0;
}

// ---- phase 4: V = I + W, J-orthogonalized in FP64 ---------------------------------------------
template <int KM>
struct alignas(16) PivotOrth {
  static constexpr int LDV = KM + 1;   // FP64 W stride
  static constexpr int LDD = KM + 8;   // digit rows of W (halves): 16-byte aligned, ldmatrix conflict-free
  static constexpr int LDS = KM + 4;   // rows of S = fp32(J M) (floats; 16-byte aligned)
  static constexpr int NT = 4 * KM;    // threads: one warp per 8 columns
  double V[KM * LDV];                  // W = V - I, FP64, column-major
  float S[KM * LDS];                   // S[x LDS + j] = fp32((J M)[x][j])
  int dexp[KM];                        // bound exponent of column c of W (digit products)
  float red_f[NT / 32][2];
  union {
    __half D[OZ_T][KM][LDD];           // digits of W by column (digit products)
    double M[KM * LDV];                // FP64 residual (FP64 mma products)
  };
};

template <int KM>
__device__ __forceinline__ float block_max_f(float v, PivotOrth<KM>& so, int slot) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  v = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));  // v >= 0
  if (lane == 0) so.red_f[warp][slot] = v;
  __syncthreads();
  float r = 0.0f;
#pragma unroll
  for (int w = 0; w < PivotOrth<KM>::NT / 32; ++w) r = fmaxf(r, so.red_f[w][slot]);
  __syncthreads();
  return r;
}

// J-orthogonality residual M = V^T J V - J = W^T J + J W + W^T J W from digit products (ozaki.cuh).
// The linear terms are exact; W^T J W, of size |W|^2, runs on the digit path with the columns of W
// (over the k rows) as scale groups and J_r applied to the A digits by their sign bit.  So M is
// accurate to ~2^-53 |W|^2 + 2^-53 |W|, where the FP64 product V^T J V carries ~2^-53 |V|^2.
// Writes S = fp32(J M) (zero outside k x k) and returns this thread's max |M_ij|.  Warp w prepares
// columns 8w..8w+7.
template <int KM>
__device__ float oz_residual(PivotOrth<KM>& so, const int* jphys, int k, int KP) {
  constexpr int NW = PivotOrth<KM>::NT / 32, LDV = PivotOrth<KM>::LDV, LDS = PivotOrth<KM>::LDS;
  static_assert(NW * 8 == KM, "one warp per 8 columns");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  // ---- column bounds and digits; lane: rows 2 lane, 2 lane + 1 (KM = 32: the row lane)
#pragma unroll
  for (int cc = 0; cc < 8; ++cc) {
    const int c = 8 * warp + cc;
    if constexpr (KM == 64) {
      const double x0 = so.V[c * LDV + 2 * lane], x1 = so.V[c * LDV + 2 * lane + 1];
      const int ec = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(oz_bexp(x0), oz_bexp(x1)));
      unsigned d[OZ_T];
      oz_split2(oz_biased(x0, oz_bexp(x0) - ec), oz_biased(x1, oz_bexp(x1) - ec), d);
#pragma unroll
      for (int t = 0; t < OZ_T; ++t) *reinterpret_cast<unsigned*>(&so.D[t][c][2 * lane]) = d[t];
      if (lane == 0) so.dexp[c] = ec;
    } else {
      const double x0 = so.V[c * LDV + lane];
      const int ec = (int)__reduce_max_sync(0xffffffffu, (unsigned)oz_bexp(x0));
      unsigned d[OZ_T];
      oz_split2(oz_biased(x0, oz_bexp(x0) - ec), OZ_BIAS, d);
#pragma unroll
      for (int t = 0; t < OZ_T; ++t) so.D[t][c][lane] = __ushort_as_half((unsigned short)d[t]);
      if (lane == 0) so.dexp[c] = ec;
    }
  }
  __syncthreads();
  // ---- upper 16 x 8 tiles of W^T J W, then M and S
  float mloc = 0.0f;
  const int ntj = KP / 8, ntiles = (KP / 16) * ntj;
  int nth = 0;  // tiles on or above the diagonal, dealt to the warps in turn
  for (int tile = 0; tile < ntiles; ++tile) {
    const int ti = tile / ntj, tj = tile - ti * ntj;
    if (8 * tj + 7 < 16 * ti) continue;
    if (nth++ % NW != warp) continue;
    float acc[OZ_T][4];
#pragma unroll
    for (int L = 0; L < OZ_T; ++L)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[L][v] = 0.0f;
    const int arow = 16 * ti + (lane & 7) + 8 * ((lane >> 3) & 1), akof = 8 * (lane >> 4);
    const int brow = 8 * tj + (lane & 7), bkof = 8 * ((lane >> 3) & 1);
    for (int kk = 0; kk < KP; kk += 16) {
      const int r0 = kk + 2 * t4;
      const unsigned slo = (jphys[r0] < 0 ? 0x8000u : 0u) | (jphys[r0 + 1] < 0 ? 0x80000000u : 0u);
      const unsigned shi = (jphys[r0 + 8] < 0 ? 0x8000u : 0u) | (jphys[r0 + 9] < 0 ? 0x80000000u : 0u);
      unsigned fa[OZ_T][4], fb[OZ_T][2];
#pragma unroll
      for (int t = 0; t < OZ_T; ++t) {
        oz_ldsm4(fa[t], &so.D[t][arow][kk + akof]);
        fa[t][0] ^= slo;
        fa[t][1] ^= slo;
        fa[t][2] ^= shi;
        fa[t][3] ^= shi;
        oz_ldsm2(fb[t][0], fb[t][1], &so.D[t][brow][kk + bkof]);
      }
      oz_levels(acc, fa, fb);
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int x = 16 * ti + g + 8 * (v >> 1), j = 8 * tj + 2 * t4 + (v & 1);
      if (j < x) continue;  // (x, j), j >= x, covers the block; (j, x) is its mirror
      float sxj = 0.0f, sjx = 0.0f;
      if (x < k && j < k) {
        const bool nx = jphys[x] < 0, nj = jphys[j] < 0;
        int q[OZ_T];
#pragma unroll
        for (int L = 0; L < OZ_T; ++L) q[L] = f32_small_int(acc[L][v]);
        const long long hi = (long long)(q[0] * 128 + q[1]) * 16384 + (q[2] * 128 + q[3]);
        const long long lo = (long long)(q[4] * 128 + q[5]) * 16384 + (q[6] * 128 + q[7]);
        // M_xj = (W^T J W)_xj + j_j W[j][x] + j_x W[x][j]
        const float f = oz_residual_entry(hi, lo, so.dexp[x] + so.dexp[j] - 2056 - 49, oz_neg_if(so.V[x * LDV + j], nj),
                                          oz_neg_if(so.V[j * LDV + x], nx));
        mloc = fmaxf(mloc, fabsf(f));
        sxj = nx ? -f : f;  // (J M)[x][j]
        sjx = nj ? -f : f;  // (J M)[j][x]
      }
      so.S[x * LDS + j] = sxj;
      so.S[j * LDS + x] = sjx;
    }
  }
  return mloc;
}

// Phase 4 of one pair, run by all 4 KM threads of a CTA on W (Wf, column c at c LDW, k valid columns):
// true (uniform) when V is J-unitary to FP64 accuracy, with W in so.V.
template <int KM>
__device__ __forceinline__ bool pivot_orth(PivotOrth<KM>& so, float* Wf, const int* jphys, int k, int oz, int& ns) {
  using SO = PivotOrth<KM>;
  constexpr int NT = SO::NT, NW = NT / 32, LDV = SO::LDV, LDS = SO::LDS, LDW = PivotDim<KM>::LDW;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int KP = (k + 15) & ~15;
  float wm = 0.0f;
#pragma unroll
  for (int u = 0; u < KM * KM / NT; ++u) {
    const int e = tid + u * NT, r = e % KM, c = e / KM;
    const bool in = r < k && c < k;
    const float w = in ? Wf[c * LDW + r] : 0.0f;
    so.V[c * LDV + r] = oz_f2d(w);  // integer conversion: FP64 instructions are scarce on GB300
    if (!in) Wf[c * LDW + r] = 0.0f;
    wm = fmaxf(wm, fabsf(w));
  }
  wm = block_max_f<KM>(wm, so, 1);  // includes the barrier after the loop
  const bool small_w = wm <= 9.5367431640625e-7f;  // 2^-20
  // products of the FP32 columns: thread (rg, cg) takes a 4 x CB block, rows 4 rg.. , columns cg + CGN c
  constexpr int RG = KM / 4, CGN = NT / RG, CB = KM / CGN;
  static_assert(RG * CGN == NT && CGN * CB == KM, "correction blocking");
  const int rg = tid % RG, cg = tid / RG;
  ns = 0;
  for (int it = 0; it < 3; ++it) {
    // residual M = V^T J V - J, J = diag(jphys) on rows and columns
    float mloc = 0.0f;
    if (it == 0 && small_w) {
      // M = W^T J + J W + W^T J W.  The linear part is exact in FP32 when it cancels (Sterbenz)
      // and rounds relative to itself otherwise; the quadratic part is at most k 2^-40 and
      // carries FP32 relative error.  Stored as fp32(J M) directly.
      float quad[4][CB];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < CB; ++c) quad[i][c] = 0.0f;
      for (int r = 0; r < k; ++r) {
        float xv[4], jv[CB];
        const float sg = (float)jphys[r];
#pragma unroll
        for (int i = 0; i < 4; ++i) xv[i] = Wf[(4 * rg + i) * LDW + r] * sg;
#pragma unroll
        for (int c = 0; c < CB; ++c) jv[c] = Wf[(cg + CGN * c) * LDW + r];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < CB; ++c) quad[i][c] = fmaf(xv[i], jv[c], quad[i][c]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          const int x = 4 * rg + i, j = cg + CGN * c;
          float mv = 0.0f;
          if (x < k && j < k) {
            const float jx = (float)jphys[x], jj = (float)jphys[j];
            mv = (Wf[x * LDW + j] * jj + jx * Wf[j * LDW + x]) + quad[i][c];
            so.S[x * LDS + j] = jx * mv;  // (J M)[x][j]
          } else {
            so.S[x * LDS + j] = 0.0f;
          }
          mloc = fmaxf(mloc, fabsf(mv));
        }
    } else if (oz) {
      mloc = oz_residual<KM>(so, jphys, k, KP);
    } else {
      // FP64 mma, upper tiles (8 tj + 7 >= 16 ti) and the mirror of the strict lower part
      const int g = lane >> 2, t = lane & 3;
      const int ntj = KP / 8, ntiles = (KP / 16) * ntj;
      for (int tile = warp; tile < ntiles; tile += NW) {
        const int ti = tile / ntj, tj = tile % ntj;
        if (8 * tj + 7 < 16 * ti) continue;
        double c4[4] = {0.0, 0.0, 0.0, 0.0};
        for (int kq = 0; kq < KP; kq += 16) {
          double av[8], bv[4];
#pragma unroll
          for (int u = 0; u < 8; ++u) av[u] = so.V[(16 * ti + g + 8 * (u & 1)) * LDV + kq + 4 * t + (u >> 1)];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = kq + 4 * t + u;
            bv[u] = oz_neg_if(so.V[(8 * tj + g) * LDV + r], jphys[r] < 0);
          }
          dmma16816(c4, av, bv);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = 16 * ti + g + 8 * (u >> 1), j = 8 * tj + 2 * t + (u & 1);
          if (j < i) continue;  // written once, from the tile holding (j, i) ... (i, j), j >= i
          const double v = c4[u] + (oz_neg_if(so.V[i * LDV + j], jphys[j] < 0) + oz_neg_if(so.V[j * LDV + i], jphys[i] < 0));
          so.M[j * LDV + i] = v;
          so.M[i * LDV + j] = v;
        }
      }
      __syncthreads();
      for (int e = tid; e < KP * KP; e += NT) {
        const int x = e % KP, j = e / KP;
        const double mv = (x < k && j < k) ? so.M[j * LDV + x] : 0.0;
        mloc = fmaxf(mloc, (float)fabs(mv));
        so.S[x * LDS + j] = (float)oz_neg_if(mv, jphys[x] < 0);
      }
    }
    const float mm = block_max_f<KM>(mloc, so, 0);
    if (mm <= 4.0e-16f) return true;
    // V <- V - V (J M) / 2 = V - (S + W S) / 2: the correction is O(|M|), formed in FP32 from the
    // FP32 columns; the FP32 columns follow in FP32
    f2 sum[2][CB];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const int r = 4 * rg + 2 * i, j = cg + CGN * c;
        sum[i][c] = f2_make(so.S[r * LDS + j], so.S[(r + 1) * LDS + j]);
      }
    for (int x = 0; x < k; ++x) {
      const ulonglong2 wv = *reinterpret_cast<const ulonglong2*>(&Wf[x * LDW + 4 * rg]);
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const float sv = so.S[x * LDS + cg + CGN * c];
        const f2 s2 = f2_make(sv, sv);
        sum[0][c] = f2_fma(wv.x, s2, sum[0][c]);
        sum[1][c] = f2_fma(wv.y, s2, sum[1][c]);
      }
    }
    __syncthreads();  // every read of Wf done
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const int j = cg + CGN * c;
      if (j >= k) continue;
      const float h[4] = {f2_lo(sum[0][c]), f2_hi(sum[0][c]), f2_lo(sum[1][c]), f2_hi(sum[1][c])};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 4 * rg + i;
        if (r < k) {
          so.V[j * LDV + r] -= oz_f2d(0.5f * h[i]);
          Wf[j * LDW + r] -= 0.5f * h[i];
        }
      }
    }
    ++ns;
    __syncthreads();
    // predicted residual after this step: quadratic term + FP32 rounding of the correction
    if (mm * mm + 1.0e-6f * mm <= 2.0e-16f) return true;
  }
  return false;
}

// What the core leaves for the other kernels of the step when the pivot's phases run apart: in the
// pair's V_P buffer (KM x KM doubles), W in FP32, then the orders and signs.
template <int KM>
struct PivotHandoff {
  float W[KM * PivotDim<KM>::LDW];
  int perm[KM], linv[KM], jphys[KM];
  static_assert((KM * PivotDim<KM>::LDW + 3 * KM) * 4 <= KM * KM * 8, "fits the V_P buffer");
};

// V_P = P V Pi: V_P[perm[r]][linv[c]] = V[r][c], FP64
template <int KM, class F>
__device__ __forceinline__ void write_vp(const JacProb& a, int pair, int k, const int* perm, const int* linv, int nt, F v) {
  double* out = a.vp + (size_t)pair * a.apld * a.apld;
  for (int e = threadIdx.x; e < KM * KM; e += nt) {
    const int r = e % KM, c = e / KM;
    if (r < k && c < k) out[(size_t)linv[c] * a.apld + perm[r]] = v(r, c);
  }
}

template <int KM>
struct PivotSmem {  // ORTH kernels; the core alone needs st, work and Wf
  PivotState<KM> st;
  float Wf[KM * PivotDim<KM>::LDW];
  union {
    PivotWork<KM> work;
    PivotOrth<KM> orth;
  };
};
template <int KM>
constexpr size_t core_smem_bytes() {
  return offsetof(PivotSmem<KM>, work) + sizeof(PivotWork<KM>);
}

__device__ __forceinline__ bool in_step(const JacProb& a, int s, int pair) {
  return a.active && s < a.nsteps && pair < a.counts[s];
}

// Modes of the pivot kernel.  PV_FULL: phases 1-4 in one CTA (FP64 sweeps).  PV_CORE: phases 1-3,
// V_P in FP64 storage from the FP32 transform (FP32 sweeps).  PV_SPLIT: phases 1-3, W handed to
// k_pivot_orth: the core needs less than half the shared memory of phase 4, so three pivots run on an
// SM while phase 4 takes the SM for a short time only (many pivots per step).  4000 problems of
// orders 8..128, all pivots of a sweep step: 1.24 ms, against 4.1 ms with one 212 KB CTA per SM.
// MINB: blocks per SM that the registers must allow.  The 80 registers of three (KM = 32: six) cost the
// core 5 of its 73 thousand clocks for a 64-column block in a block-oriented step (order 512, mixed
// precision: 14.8 ms; with 142 registers 14.4), so steps with no more pivots than SMs take all they need.
enum { PV_FULL = 0, PV_CORE = 1, PV_SPLIT = 2 };
constexpr int many_blocks(int km) { return km == 32 ? 6 : 3; }

template <int KM, int MODE, int MINB>
__global__ void __launch_bounds__(4 * KM, MINB)
    k_pivot(const JacProb* __restrict__ probs, int s, PivotParams pp) {
  extern __shared__ __align__(16) unsigned char pv_raw[];
  PivotSmem<KM>& sm = *reinterpret_cast<PivotSmem<KM>*>(pv_raw);
  const JacProb& a = probs[blockIdx.y];
  const int pair = blockIdx.x, tid = threadIdx.x;
  if (!in_step(a, s, pair) || pair_skip_known(a, s, pair)) return;
  PairStat* stats = a.stats + (size_t)s * a.half;
  if constexpr (MODE != PV_FULL) {
    if (pivot_core<KM, false>(sm.st, sm.work, nullptr, sm.Wf, a, s, pair, pp) != 0) return;
    __syncthreads();
    const int k = sm.st.k;
    if constexpr (MODE == PV_CORE) {
      write_vp<KM>(a, pair, k, sm.st.perm, sm.st.linv, 4 * KM, [&](int r, int c) {
        const float w = sm.Wf[c * PivotDim<KM>::LDW + r];
        return r == c ? oz_f2d(w) + 1.0 : oz_f2d(w);
      });
    } else {
      PivotHandoff<KM>& h = *reinterpret_cast<PivotHandoff<KM>*>(a.vp + (size_t)pair * a.apld * a.apld);
      for (int e = tid; e < k * PivotDim<KM>::LDW / 4; e += 4 * KM)
        reinterpret_cast<float4*>(h.W)[e] = reinterpret_cast<const float4*>(sm.Wf)[e];
      if (tid < KM) {
        h.perm[tid] = sm.st.perm[tid];
        h.linv[tid] = sm.st.linv[tid];
        h.jphys[tid] = sm.st.jphys[tid];
      }
    }
    if (tid == 0) {
      a.skip[pair] = 0;
      if (MODE == PV_CORE) pair_record(a, s, pair, true);
      stats[pair] = sm.st.st;
    }
  } else {
    if (pivot_core<KM, false>(sm.st, sm.work, nullptr, sm.Wf, a, s, pair, pp) != 0) return;
    __syncthreads();
    const int k = sm.st.k;
    int ns = 0;
    const bool ok = pivot_orth<KM>(sm.orth, sm.Wf, sm.st.jphys, k, pp.oz, ns);
    if (ok)
      write_vp<KM>(a, pair, k, sm.st.perm, sm.st.linv, 4 * KM, [&](int r, int c) {
        const double w = sm.orth.V[c * PivotOrth<KM>::LDV + r];
        return r == c ? w + 1.0 : w;
      });
    if (tid == 0) {
      // not J-unitary to FP64 accuracy after the step budget: FP64 pivot kernel
      a.skip[pair] = ok ? 0 : 2;
      if (!ok) atomicOr(a.pflags, JAC_DEVERR_HANDOVER);
      else pair_record(a, s, pair, true);
      sm.st.st.ns_steps = ns;
      sm.st.st.cyc[3] = clock64() - sm.st.t_core;
      stats[pair] = sm.st.st;
    }
  }
}

// Phase 4 of the pairs whose core ran in k_pivot<KM, PV_SPLIT>.  Grid and guards as the core.
template <int KM>
struct OrthSmem {
  float Wf[KM * PivotDim<KM>::LDW];
  int perm[KM], linv[KM], jphys[KM];
  PivotOrth<KM> orth;
};
template <int KM>
__global__ void __launch_bounds__(4 * KM, KM == 32 ? 4 : 1)
    k_pivot_orth(const JacProb* __restrict__ probs, int s, PivotParams pp) {
  extern __shared__ __align__(16) unsigned char pv_raw[];
  OrthSmem<KM>& sm = *reinterpret_cast<OrthSmem<KM>*>(pv_raw);
  const JacProb& a = probs[blockIdx.y];
  const int pair = blockIdx.x, tid = threadIdx.x;
  if (!in_step(a, s, pair) || a.skip[pair] != 0) return;
  const long long t0 = clock64();
  const int* sp = a.pairs + (size_t)s * a.half * 2;
  const int p = sp[2 * pair], q = sp[2 * pair + 1];
  const int k = a.boff[p + 1] - a.boff[p] + a.boff[q + 1] - a.boff[q];
  const PivotHandoff<KM>& h = *reinterpret_cast<const PivotHandoff<KM>*>(a.vp + (size_t)pair * a.apld * a.apld);
  for (int e = tid; e < k * PivotDim<KM>::LDW / 4; e += 4 * KM)
    reinterpret_cast<float4*>(sm.Wf)[e] = reinterpret_cast<const float4*>(h.W)[e];
  if (tid < KM) {
    sm.perm[tid] = h.perm[tid];
    sm.linv[tid] = h.linv[tid];
    sm.jphys[tid] = h.jphys[tid];
  }
  __syncthreads();  // the hand-over is read: V_P may take its place
  int ns = 0;
  const bool ok = pivot_orth<KM>(sm.orth, sm.Wf, sm.jphys, k, pp.oz, ns);
  if (ok)
    write_vp<KM>(a, pair, k, sm.perm, sm.linv, 4 * KM, [&](int r, int c) {
      const double w = sm.orth.V[c * PivotOrth<KM>::LDV + r];
      return r == c ? w + 1.0 : w;
    });
  if (tid == 0) {
    if (!ok) {
      a.skip[pair] = 2;
      atomicOr(a.pflags, JAC_DEVERR_HANDOVER);
    } else {
      pair_record(a, s, pair, true);
    }
    PairStat& st = a.stats[(size_t)s * a.half + pair];
    st.ns_steps = ns;
    st.cyc[3] = clock64() - t0;
  }
}

// ---- the fused step kernel ---------------------------------------------------------------------
// One step of the FP32 sweeps for one pair in one CTA: the Gram block, the pivot and the block
// update, with X_P = [G_p G_q] read from global memory once and written once.  The m rows of X_P
// stay in shared memory from the Gram to the update; the rows of V go through the pivot's work area
// in chunks of 64.  Used when every problem of the launch has m <= fused_step_max_rows(KM).  The
// launch asks for the shared memory of its largest m, so several CTAs share an SM.
template <int KM>
struct FusedLayout {
  static constexpr int LDX = KM + 4;  // staged rows of X_P (floats; 16-byte aligned rows)
  static constexpr int LDB = KM + 4;  // V_P in FP32, row c = input column
  static constexpr int MF = KM == 32 ? 96 : 192;  // largest m
  // Bs, then the chunk of V, over the pivot's work area
  static constexpr int WORK = (int)sizeof(PivotWork<KM>) / 4 > KM * LDB + 64 * LDX ? (int)sizeof(PivotWork<KM>) / 4
                                                                                   : KM * LDB + 64 * LDX;
  struct Smem {
    PivotState<KM> st;
    float Wf[KM * PivotDim<KM>::LDW];  // A_P in FP32, then W
    alignas(16) float work[WORK];
    alignas(16) float X[1];            // [r][c], m rows
  };
  static constexpr size_t bytes(int m) { return offsetof(Smem, X) + (size_t)m * LDX * 4; }
};

template <int KM>
__global__ void __launch_bounds__(4 * KM, KM == 32 ? 4 : 2)
    k_step_fused(const JacProb* __restrict__ probs, int s, PivotParams pp, int mmax) {
  using FL = FusedLayout<KM>;
  constexpr int NT = 4 * KM, LDX = FL::LDX, LDB = FL::LDB, LDW = PivotDim<KM>::LDW;
  constexpr int CT = KM / 4;  // 4-column groups
  static_assert(NT / CT == 16, "16 row groups");
  extern __shared__ __align__(16) unsigned char pv_raw[];
  typename FL::Smem& sm = *reinterpret_cast<typename FL::Smem*>(pv_raw);
  const JacProb& a = probs[blockIdx.y];
  const int pair = blockIdx.x;
  if (!in_step(a, s, pair) || pair_skip_known(a, s, pair)) return;
  const int tid = threadIdx.x, tx = tid % CT, ty = tid / CT;
  const int* sp = a.pairs + (size_t)s * a.half * 2;
  const int p = sp[2 * pair], q = sp[2 * pair + 1];
  const int op = a.boff[p], wp = a.boff[p + 1] - op, oq = a.boff[q], wq = a.boff[q + 1] - oq;
  const int k = wp + wq, m = a.mp;
  // the driver launches this kernel for the FP32 sweeps within these bounds; anything else is
  // reported, never trapped
  if (k > KM || m > mmax || pp.ns_mode) {
    if (tid == 0) {
      atomicOr(a.pflags, JAC_DEVERR_INNER_LIMIT);
      a.skip[pair] = 1;
    }
    return;
  }
  auto pcol = [&](int c) { return c < wp ? op + c : oq + (c - wp); };
  float* Xs = sm.X;                  // [r][c], m rows
  float* Bs = sm.work;               // [c][j]
  float* Vst = sm.work + KM * LDB;   // 64-row chunk of V, [r][c]

  // ---- 0. X_P into shared memory (zero columns beyond k); A_P = X_P^T X_P in FP32
  {
    const int nw = NT / 32, warp = tid >> 5, lane = tid & 31;
    for (int c = warp; c < KM; c += nw) {  // a warp per column, consecutive lanes consecutive rows
      const float* col = a.G32 + (size_t)pcol(c < k ? c : 0) * a.mp;
      for (int rr = 0; rr < m; rr += 32 * 6) {
        float v[6];
#pragma unroll
        for (int u = 0; u < 6; ++u) {
          const int r = rr + lane + 32 * u;
          v[u] = (c < k && r < m) ? __ldg(col + r) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 6; ++u) {
          const int r = rr + lane + 32 * u;
          if (r < m) Xs[r * LDX + c] = v[u];
        }
      }
    }
  }
  __syncthreads();
  {
    // thread (ty, tx): rows RPT ty .. RPT ty + RPT - 1 and columns 4 tx .. 4 tx + 3 of A_P; the
    // entries (i, j) and (j, i) take the same products in the same order (exactly symmetric)
    constexpr int RPT = KM / 16;
    f2 acc[RPT][2];
#pragma unroll
    for (int u = 0; u < RPT; ++u) acc[u][0] = acc[u][1] = f2_make(0.0f, 0.0f);
#pragma unroll 4
    for (int r = 0; r < m; ++r) {
      const float* xr = Xs + r * LDX;
      const ulonglong2 xj = *reinterpret_cast<const ulonglong2*>(xr + 4 * tx);
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        const float xi = xr[RPT * ty + u];
        const f2 x2 = f2_make(xi, xi);
        acc[u][0] = f2_fma(x2, xj.x, acc[u][0]);
        acc[u][1] = f2_fma(x2, xj.y, acc[u][1]);
      }
    }
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      const int i = RPT * ty + u;
      sm.Wf[(4 * tx) * LDW + i] = f2_lo(acc[u][0]);
      sm.Wf[(4 * tx + 1) * LDW + i] = f2_hi(acc[u][0]);
      sm.Wf[(4 * tx + 2) * LDW + i] = f2_lo(acc[u][1]);
      sm.Wf[(4 * tx + 3) * LDW + i] = f2_hi(acc[u][1]);
    }
  }
  __syncthreads();

  // ---- 1.-3. the pivot
  const int pr = pivot_core<KM, true>(sm.st, *reinterpret_cast<PivotWork<KM>*>(sm.work), sm.Wf, sm.Wf, a, s, pair, pp);
  __syncthreads();
  if (pr == 2) {
    // handed over: the FP64 pivot kernel reads A_P from the Gram output, as after the Gram kernel
    double* A = a.Ap + (size_t)pair * a.apld * a.apld;
    for (int e = tid; e < k * k; e += NT) A[(e / k) * a.apld + e % k] = oz_f2d(sm.Wf[(e / k) * LDW + e % k]);
  }
  if (pr != 0) return;

  // ---- 4. [X_P; V rows] <- [X_P; V rows] V_P in FP32, V_P[perm[r]][linv[c]] = V[r][c]
  for (int e = tid; e < KM * KM; e += NT) {
    const int r = e % KM, c = e / KM;
    if (r < k && c < k) Bs[sm.st.perm[r] * LDB + sm.st.linv[c]] = sm.Wf[c * LDW + r] + (r == c ? 1.0f : 0.0f);
  }
  if (tid == 0) {
    a.skip[pair] = 3;  // updated by this kernel itself
    pair_record(a, s, pair, true);
    a.stats[(size_t)s * a.half + pair] = sm.st.st;
  }
  __syncthreads();
  // thread (ty, tx): rows 4 ty .. 4 ty + 3 of a 64-row chunk, columns 4 tx .. 4 tx + 3
  auto update_chunk = [&](const float* X, int rows, float* dst, int ld, int r0) {
    f2 acc[4][2];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u][0] = acc[u][1] = f2_make(0.0f, 0.0f);
    if (4 * ty < rows) {
#pragma unroll 4
      for (int c = 0; c < k; ++c) {
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(Bs + c * LDB + 4 * tx);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float x = X[(4 * ty + u) * LDX + c];
          const f2 x2 = f2_make(x, x);
          acc[u][0] = f2_fma(x2, b.x, acc[u][0]);
          acc[u][1] = f2_fma(x2, b.y, acc[u][1]);
        }
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int j = 4 * tx + v;
        if (j >= k) continue;
        float* col = dst + (size_t)pcol(j) * ld + r0 + 4 * ty;  // rows are a multiple of 16
        float o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) o[u] = (v & 1) ? f2_hi(acc[u][v >> 1]) : f2_lo(acc[u][v >> 1]);
        *reinterpret_cast<float4*>(col) = make_float4(o[0], o[1], o[2], o[3]);
      }
    }
  };
  for (int r0 = 0; r0 < m; r0 += 64) update_chunk(Xs + r0 * LDX, min(64, m - r0), a.G32, a.mp, r0);
  if (a.V32) {
    for (int r0 = 0; r0 < a.np; r0 += 64) {
      const int rows = min(64, a.np - r0);
      constexpr int NV = KM * 64 / NT;
      float v[NV];
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int e = u * NT + tid, c = e / 64, r = e % 64;
        v[u] = (c < k && r < rows) ? a.V32[(size_t)pcol(c) * a.np + r0 + r] : 0.0f;
      }
      __syncthreads();  // the previous chunk's reads of Vst are done
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int e = u * NT + tid;
        Vst[(e % 64) * LDX + e / 64] = v[u];
      }
      __syncthreads();
      update_chunk(Vst, rows, a.V32, a.np, r0);
    }
  }
}

int fused_step_max_rows(int km) { return km == 32 ? FusedLayout<32>::MF : FusedLayout<64>::MF; }

static_assert(sizeof(PivotSmem<64>) <= 232448, "pivot shared memory above the 227 KB per-CTA limit");

// Host side of the instantiations (a kernel template is launched from its own translation unit).
template <int KM>
static bool set_attributes() {
  auto set = [](auto kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
  };
  bool ok = set(k_pivot<KM, PV_FULL, 1>, sizeof(PivotSmem<KM>));
  ok &= set(k_pivot<KM, PV_CORE, 1>, core_smem_bytes<KM>());
  ok &= set(k_pivot<KM, PV_CORE, many_blocks(KM)>, core_smem_bytes<KM>());
  ok &= set(k_pivot<KM, PV_SPLIT, many_blocks(KM)>, core_smem_bytes<KM>());
  ok &= set(k_pivot_orth<KM>, sizeof(OrthSmem<KM>));
  ok &= set(k_step_fused<KM>, FusedLayout<KM>::bytes(FusedLayout<KM>::MF));
  return ok;
}
int pivot_set_attributes() { return set_attributes<32>() && set_attributes<64>() ? 0 : 1; }

// Grid (max_half, nprob): one CTA per pivot block.  Returns the number of kernels launched.
// FP64 sweeps with more pivots in the step than SMs run the core and phase 4 as two kernels.
constexpr int kSplitPivots = 152;

template <int KM>
static int launch_pivot(int max_half, int nprob, cudaStream_t st, const JacProb* probs, int s, const PivotParams& pp) {
  const dim3 grid(max_half, nprob);
  const bool few = (long long)max_half * nprob <= kSplitPivots;
  if (!pp.ns_mode) {
    if (few) k_pivot<KM, PV_CORE, 1><<<grid, 4 * KM, core_smem_bytes<KM>(), st>>>(probs, s, pp);
    else k_pivot<KM, PV_CORE, many_blocks(KM)><<<grid, 4 * KM, core_smem_bytes<KM>(), st>>>(probs, s, pp);
    return 1;
  }
  if (few) {
    k_pivot<KM, PV_FULL, 1><<<grid, 4 * KM, sizeof(PivotSmem<KM>), st>>>(probs, s, pp);
    return 1;
  }
  k_pivot<KM, PV_SPLIT, many_blocks(KM)><<<grid, 4 * KM, core_smem_bytes<KM>(), st>>>(probs, s, pp);
  k_pivot_orth<KM><<<grid, 4 * KM, sizeof(OrthSmem<KM>), st>>>(probs, s, pp);
  return 2;
}
int pivot_launch(int km, int max_half, int nprob, cudaStream_t st, const JacProb* probs, int s, const PivotParams& pp) {
  return km == 32 ? launch_pivot<32>(max_half, nprob, st, probs, s, pp)
                  : launch_pivot<64>(max_half, nprob, st, probs, s, pp);
}

// Grid (max_half, nprob): one CTA per pair, the whole FP32 step; every problem has m <= mmax <=
// fused_step_max_rows(km) padded rows.
void fused_step_launch(int km, int max_half, int nprob, cudaStream_t st, const JacProb* probs, int s,
                       const PivotParams& pp, int mmax) {
  if (km == 32)
    k_step_fused<32><<<dim3(max_half, nprob), 4 * 32, FusedLayout<32>::bytes(mmax), st>>>(probs, s, pp, mmax);
  else
    k_step_fused<64><<<dim3(max_half, nprob), 4 * 64, FusedLayout<64>::bytes(mmax), st>>>(probs, s, pp, mmax);
}

}  // namespace jac
