// ozaki.cu -- the FP64 Gram (Eq. (3.4)) of a step, and a batched GEMM (the precision switch's
// V^T J V and G_in V, the backward's products), from exact FP16 tensor-core digit products
// (ozaki.cuh).  Same grids, work split and results as k_gram (gram_update.cu) and k_gemm64
// (dense.cu), to FP64 accuracy.  The digit update (Algorithm 3.4) is in tc_digits.cu.
//
// Scale groups of the Gram X^T X: the columns of X over a stage of rows (each column is one row
// of A = X^T and one column of B = X).
#include <cooperative_groups.h>

#include <mutex>

#include "jacobi_common.cuh"
#include "pair_cache.cuh"
#include "ozaki.cuh"

namespace cg = cooperative_groups;

namespace jac {

__device__ __forceinline__ int oz_pair_col(int c, int wp, int op, int oq) { return c < wp ? op + c : oq + (c - wp); }

// ------------------------------------------------------------------------------------ Gram
// Grid (half * CS, nprob), cluster (CS, 1, 1), 256 threads; the CS CTAs of a cluster split the
// rows of one pair as in k_gram.  A CTA takes its rows in stages of 128: warp w loads columns
// w, w + 8, .. (lane: rows 2 lane, 2 lane + 1, 64 + 2 lane, 65 + 2 lane), sets each column's bound
// exponent E_c over the stage, and stores the digits D[t][c][row].  The upper 16 x 8 tiles of the
// k x k block (20 at k = 64) go to the warps (at most 3 each) and are summed in FP64 across stages.
// Columns, rows and tiles past k and past the rows are not formed, a level sum is rounded without an
// FP64 instruction, and the cluster's sum adds only what is there: one block of 64 rows and 16
// columns 21.5 -> 10.4 us, 4000 problems of orders 8..128 572 -> 265 us (mma.sync is then ~half of a
// stage; blocks of many stages go to k_gram_oz_tc).
#define OZG_ROWS 128
#define OZG_NL 8  // levels kept: the Gram's groups are its own columns, bounds within ~4x of the terms
#define OZG_P (OZG_ROWS + 8)  // 272-byte digit rows: 16-byte aligned, ldmatrix conflict-free
struct OzGramSmem {
  __half D[OZ_T][JAC_KMAX][OZG_P];
  double C[JAC_KMAX][JAC_KMAX + 1];
  int E[JAC_KMAX];
};

// idx-th upper tile (8 tj + 7 >= 16 ti) of a block of ntj 8-column tiles, row by row; false past the last
__device__ __forceinline__ bool oz_upper_tile(int idx, int ntj, int& ti, int& tj) {
  for (ti = 0; 2 * ti < ntj; ++ti) {
    const int len = ntj - 2 * ti;
    if (idx < len) {
      tj = 2 * ti + idx;
      return true;
    }
    idx -= len;
  }
  return false;
}

__global__ void __launch_bounds__(256) k_gram_oz(const JacProb* __restrict__ probs, int s, int CS) {
  extern __shared__ __align__(16) unsigned char oz_raw[];
  OzGramSmem& sm = *reinterpret_cast<OzGramSmem*>(oz_raw);
  cg::cluster_group cluster = cg::this_cluster();
  const JacProb& a = probs[blockIdx.y];
  const int pair = blockIdx.x / CS;
  const int crank = (int)cluster.block_rank();
  if (!a.active || s >= a.nsteps || pair >= a.counts[s]) return;
  const int* sp = a.pairs + (size_t)s * a.half * 2;
  const int p = sp[2 * pair], q = sp[2 * pair + 1];
  if (pair_known(a, s, pair)) return;  // uniform
  const int op = a.boff[p], wp = a.boff[p + 1] - op, oq = a.boff[q], wq = a.boff[q + 1] - oq;
  const int k = wp + wq, ntj = (k + 7) >> 3;  // 8-column tiles
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
  const int rpc = ((a.mp / CS + 15) & ~15);
  const int r_begin = min(a.mp, crank * rpc), r_end = min(a.mp, r_begin + rpc);
  // columns warp, warp + 8, ... below the last 16-column tile's end; columns >= k have zero digits
  const int ncc = (((k + 15) & ~15) - warp + 7) >> 3;

  double tot[3][4];
#pragma unroll
  for (int u = 0; u < 3; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) tot[u][v] = 0.0;

  for (int r0 = r_begin; r0 < r_end; r0 += OZG_ROWS) {
    const int rs = min(OZG_ROWS, r_end - r0);  // multiple of 16
    const bool two = rs > 64;                  // rows 64.. of the stage
    // ---- load the stage (all loads first), bound exponents, digits
    double2 x[8][2];
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
      const int c = warp + 8 * cc;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = 64 * i + 2 * lane;
        x[cc][i] = (c < k && r < rs)
                       ? __ldg(reinterpret_cast<const double2*>(a.Gw + (size_t)oz_pair_col(c, wp, op, oq) * a.mp + r0 + r))
                       : make_double2(0.0, 0.0);
      }
    }
    __syncthreads();  // the previous stage's digits and exponents are no longer read
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
      if (cc >= ncc) break;
      const int c = warp + 8 * cc;
      const int e = max(max(oz_bexp(x[cc][0].x), oz_bexp(x[cc][0].y)), max(oz_bexp(x[cc][1].x), oz_bexp(x[cc][1].y)));
      const int ec = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
      if (lane == 0) sm.E[c] = ec;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (i == 1 && !two) break;
        unsigned w[OZ_T];
        oz_split2(oz_biased(x[cc][i].x, oz_bexp(x[cc][i].x) - ec), oz_biased(x[cc][i].y, oz_bexp(x[cc][i].y) - ec), w);
#pragma unroll
        for (int t = 0; t < OZ_T; ++t) *reinterpret_cast<unsigned*>(&sm.D[t][c][64 * i + 2 * lane]) = w[t];
      }
    }
    __syncthreads();
    // ---- digit products of the upper tiles
    const int kend = (rs + 15) & ~15;
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      int ti, tj;
      if (!oz_upper_tile(warp + 8 * u, ntj, ti, tj)) break;
      float acc[OZG_NL][4];
#pragma unroll
      for (int L = 0; L < OZG_NL; ++L)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[L][v] = 0.0f;
      // ldmatrix rows: A (X^T, rows = columns i of the tile) and B (X, rows = columns j)
      const int arow = 16 * ti + (lane & 7) + 8 * ((lane >> 3) & 1), akof = 8 * (lane >> 4);
      const int brow = 8 * tj + (lane & 7), bkof = 8 * ((lane >> 3) & 1);
#pragma unroll 1
      for (int kk = 0; kk < kend; kk += 16) {
        unsigned fa[OZ_T][4], fb[OZ_T][2];
#pragma unroll
        for (int t = 0; t < OZ_T; ++t) {
          oz_ldsm4(fa[t], &sm.D[t][arow][kk + akof]);
          oz_ldsm2(fb[t][0], fb[t][1], &sm.D[t][brow][kk + bkof]);
        }
        oz_levels(acc, fa, fb);
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int i = 16 * ti + g + 8 * (v >> 1), j = 8 * tj + 2 * t4 + (v & 1);
        const double y = oz_value_int(acc, v, sm.E[i] + sm.E[j] - 2056);
        tot[u][v] = (r0 == r_begin) ? y : tot[u][v] + y;
      }
    }
  }
  double* out = a.Ap + (size_t)pair * a.apld * a.apld;
  if (CS == 1) {  // nothing to add up: (i, j), j >= i, and its mirror
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      int ti, tj;
      if (!oz_upper_tile(warp + 8 * u, ntj, ti, tj)) break;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int i = 16 * ti + g + 8 * (v >> 1), j = 8 * tj + 2 * t4 + (v & 1);
        if (j >= i && j < k) {
          out[j * a.apld + i] = tot[u][v];
          out[i * a.apld + j] = tot[u][v];
        }
      }
    }
    return;
  }
  // ---- partial -> own shared memory: (i, j), j >= i
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    int ti, tj;
    if (!oz_upper_tile(warp + 8 * u, ntj, ti, tj)) break;
#pragma unroll
    for (int v = 0; v < 4; ++v) sm.C[16 * ti + g + 8 * (v >> 1)][8 * tj + 2 * t4 + (v & 1)] = tot[u][v];
  }
  cluster.sync();
  // the upper triangle, rows n and k - 1 - n together as one row of k + 1 entries; only the CS - 1
  // additions that are needed (an FP64 addition costs the SM 20 clocks per warp: sixteen for every
  // entry of the full block, most of them of zeros, were a third of a single-stage Gram)
  const int totn = ((k + 1) >> 1) * (k + 1), per = (totn + CS - 1) / CS;
  const int e0 = crank * per, e1 = min(totn, e0 + per);
  for (int e = e0 + tid; e < e1; e += 256) {
    const int n = e / (k + 1), o = e - n * (k + 1);
    int i = n, j = n + o;
    if (j >= k) {
      i = k - 1 - n;
      j = i + (o - (k - n));
      if (i == n) continue;  // the middle row of an odd block
    }
    double part[16];  // all remote loads issued before the fixed-order sum
#pragma unroll
    for (int rk = 0; rk < 16; ++rk)
      part[rk] = (rk < CS) ? cluster.map_shared_rank(&sm.C[0][0], rk)[i * (JAC_KMAX + 1) + j] : 0.0;
    double sum = part[0];
#pragma unroll
    for (int rk = 1; rk < 16; ++rk)
      if (rk < CS) sum += part[rk];
    out[j * a.apld + i] = sum;
    out[i * a.apld + j] = sum;
  }
  cluster.sync();  // keep every partial alive until all remote reads are done
}

#define OZ_NO_EXP (-100000)

size_t oz_gram_smem_bytes() { return sizeof(OzGramSmem); }

// ------------------------------------------------------------------------------- GEMM
// C = op(A) diag(sb) op(B) - diag(dsub), the contract of k_gemm64 (dense.cu), from FP16 digit
// products: column-major, C is Mr x Nc, batch member blockIdx.z at element strides sa, sbb, sc;
//   transA = 1: op(A)[i][r] = A[i * lda + r], else A[r * lda + i];
//   transB = 1: op(B)[r][j] = B[r * ldb + j], else B[j * ldb + r];
//   sb: optional +-1 per r; dsub: optional, its sign subtracted on the diagonal;
//   sym = 1: C symmetric (Mr == Nc), entries j >= i computed and mirrored.
// K runs in segments of 256 (4 chunks of 64), each an exact FP32 level sum recombined into FP64.
// Per segment the scales are those of the digit update (tc_digits.cu): c_r = bound exponent of column r of the CTA's
// op(A) rows, then the rows of op(A) D^-1 and the columns of D op(B) (D = diag(2^c_r)) are the
// scale groups, so a term is exact to 2^-53 of its own row and column sizes even when the columns
// of A (or rows of B) are graded.  Two CTAs per SM (112 KB each): the digits of one are made while
// the other multiplies; with integer rounding and coalesced column bounds the adjoint of 256 problems
// of order 256 takes 4.71 ms instead of 6.62.  Grid (ceil(Mr/64), ceil(Nc/32), batch), 256 threads: warp w
// computes row tile w & 3 (16 rows) and column tiles 2 (w >> 2) + {0, 1}.
#define OZM_TI 64
#define OZM_TJ 32
#define OZM_KC 64
#define OZM_SEG 256
#define OZM_P (OZM_KC + 8)
#define OZM_NL 9
struct OzGemmSmem {
  __half A[OZ_T][OZM_TI][OZM_P];  // digits of op(A) D^-1: [t][row][r]
  __half B[OZ_T][OZM_TJ][OZM_P];  // digits of D op(B): [t][column][r]
  int ck[OZM_SEG];                // c_r of the segment (0: zero column)
  int rexp[OZM_TI];
  int cexp[OZM_TJ];
};

__global__ void __launch_bounds__(256, 2) k_gemm_oz(int Mr, int Nc, int K, const double* __restrict__ A, int lda,
                                                int transA, const double* __restrict__ B, int ldb,
                                                const int8_t* __restrict__ sb, const int8_t* __restrict__ dsub,
                                                double* __restrict__ C, int ldc, int sym, int transB, long long sa,
                                                long long sbb, long long sc) {
  extern __shared__ __align__(16) unsigned char oz_raw[];
  OzGemmSmem& sm = *reinterpret_cast<OzGemmSmem*>(oz_raw);
  A += (size_t)blockIdx.z * sa;
  B += (size_t)blockIdx.z * sbb;
  C += (size_t)blockIdx.z * sc;
  const int i0 = blockIdx.x * OZM_TI, j0 = blockIdx.y * OZM_TJ;
  if (sym && j0 + OZM_TJ - 1 < i0) return;  // no entry with j >= i
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
  const int ai = tid >> 2, ar = tid & 3, bj = tid >> 3, br = tid & 7;  // 4 threads per row, 8 per column
  const bool rowok = i0 + ai < Mr, colok = j0 + bj < Nc;
  const int ti = warp & 3, tj0 = 2 * (warp >> 2);
  const int arow = 16 * ti + (lane & 7) + 8 * ((lane >> 3) & 1), akof = 8 * (lane >> 4);
  const int bcol = 8 * tj0 + (lane & 7), bkof = 8 * ((lane >> 3) & 1);
  auto a_at = [&](int i, int r) -> double {  // op(A)[i0 + i][r], in range
    return transA ? A[(size_t)(i0 + i) * lda + r] : A[(size_t)r * lda + i0 + i];
  };
  auto b_at = [&](int j, int r) -> double {  // op(B)[r][j0 + j] with the sign sb_r, in range
    const double y = transB ? B[(size_t)r * ldb + j0 + j] : B[(size_t)(j0 + j) * ldb + r];
    return (sb && sb[r] < 0) ? oz_neg_if(y, true) : y;
  };
  float acc0[OZM_NL][4], acc1[OZM_NL][4];
  double res[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int e = 0; e < 4; ++e) res[h][e] = 0.0;
  for (int s0 = 0; s0 < K; s0 += OZM_SEG) {
    const int slen = min(OZM_SEG, K - s0);
    // ---- c_r of the CTA's op(A) rows, the lanes along the contiguous index: thread tid takes column
    // s0 + tid (rows of A contiguous in r), or warp w columns w, w + 8, ..
    __syncthreads();  // the previous segment's exponents are no longer read
    if (transA) {
      int c = 0;
      if (tid < slen) {
        const int imax = min(OZM_TI, Mr - i0);
#pragma unroll 16
        for (int i = 0; i < imax; ++i) c = max(c, oz_bexp(a_at(i, s0 + tid)));
      }
      sm.ck[tid] = c;
    } else {
#pragma unroll 8
      for (int r = warp; r < slen; r += 8) {
        const int e0 = (i0 + lane < Mr) ? oz_bexp(a_at(lane, s0 + r)) : 0;
        const int e1 = (i0 + lane + 32 < Mr) ? oz_bexp(a_at(lane + 32, s0 + r)) : 0;
        const unsigned c = __reduce_max_sync(0xffffffffu, (unsigned)max(e0, e1));
        if (lane == 0) sm.ck[r] = (int)c;
      }
    }
    __syncthreads();
    // ---- row groups of op(A) D^-1 and column groups of D op(B)
    {
      int ea = OZ_NO_EXP, eb = OZ_NO_EXP;
      if (rowok) {
#pragma unroll 16
        for (int r = ar; r < slen; r += 4) {
          const int ex = oz_bexp(a_at(ai, s0 + r));
          if (ex != 0) ea = max(ea, ex - sm.ck[r]);
        }
      }
      if (colok) {
#pragma unroll 16
        for (int r = br; r < slen; r += 8) {
          const int ex = oz_bexp(b_at(bj, s0 + r)), c = sm.ck[r];
          if (ex != 0 && c != 0) eb = max(eb, ex + c);
        }
      }
      ea = max(ea, __shfl_xor_sync(0xffffffffu, ea, 1));
      ea = max(ea, __shfl_xor_sync(0xffffffffu, ea, 2));
      eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 1));
      eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 2));
      eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 4));
      if (ar == 0) sm.rexp[ai] = ea;
      if (br == 0) sm.cexp[bj] = eb;
    }
    __syncthreads();
    const int my_ea = sm.rexp[ai], my_eb = sm.cexp[bj];
#pragma unroll
    for (int L = 0; L < OZM_NL; ++L)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc0[L][e] = 0.0f;
        acc1[L][e] = 0.0f;
      }
    for (int kc = 0; kc < slen; kc += OZM_KC) {
      // ---- digits of the chunk, A then B (the other CTA of the SM hides the loads)
      {
        double xa[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {  // pairs of neighbours: one 32-bit store per digit
          const int r = kc + 2 * ar + 8 * (u >> 1) + (u & 1);
          xa[u] = (rowok && r < slen) ? a_at(ai, s0 + r) : 0.0;
        }
        __syncthreads();  // the previous chunk's digits are consumed
#pragma unroll
        for (int u = 0; u < 16; u += 2) {
          const int rl = 2 * ar + 8 * (u >> 1), r = kc + rl;
          unsigned w[OZ_T];
          const int c0 = (r < slen) ? sm.ck[r] : 0, c1 = (r + 1 < slen) ? sm.ck[r + 1] : 0;
          oz_split2(oz_biased(xa[u], oz_bexp(xa[u]) - c0 - my_ea), oz_biased(xa[u + 1], oz_bexp(xa[u + 1]) - c1 - my_ea), w);
#pragma unroll
          for (int t = 0; t < OZ_T; ++t) *reinterpret_cast<unsigned*>(&sm.A[t][ai][rl]) = w[t];
        }
      }
      {
        double xb[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int r = kc + 2 * br + 16 * (u >> 1) + (u & 1);
          xb[u] = (colok && r < slen) ? b_at(bj, s0 + r) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          const int rl = 2 * br + 16 * (u >> 1), r = kc + rl;
          unsigned w[OZ_T];
          const int c0 = (r < slen) ? sm.ck[r] : 0, c1 = (r + 1 < slen) ? sm.ck[r + 1] : 0;
          oz_split2(c0 != 0 ? oz_biased(xb[u], oz_bexp(xb[u]) + c0 - my_eb) : OZ_BIAS,
                    c1 != 0 ? oz_biased(xb[u + 1], oz_bexp(xb[u + 1]) + c1 - my_eb) : OZ_BIAS, w);
#pragma unroll
          for (int t = 0; t < OZ_T; ++t) *reinterpret_cast<unsigned*>(&sm.B[t][bj][rl]) = w[t];
        }
      }
      __syncthreads();
      const int kend = min(OZM_KC, (slen - kc + 15) & ~15);
#pragma unroll 1
      for (int kk = 0; kk < kend; kk += 16) {
        unsigned fa[OZ_T][4], fb[OZ_T][2];
#pragma unroll
        for (int t = 0; t < OZ_T; ++t) {
          oz_ldsm4(fa[t], &sm.A[t][arow][kk + akof]);
          oz_ldsm2(fb[t][0], fb[t][1], &sm.B[t][bcol][kk + bkof]);
        }
        oz_levels(acc0, fa, fb);
#pragma unroll
        for (int t = 0; t < OZ_T; ++t) oz_ldsm2(fb[t][0], fb[t][1], &sm.B[t][bcol + 8][kk + bkof]);
        oz_levels(acc1, fa, fb);
      }
    }
    // ---- the segment's exact level sums into FP64
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int il = 16 * ti + g + 8 * (e >> 1);
      const int jl0 = 8 * tj0 + 2 * t4 + (e & 1), jl1 = jl0 + 8;
      const double y0 = oz_value9(acc0, e, sm.rexp[il] + sm.cexp[jl0] - 2056);
      const double y1 = oz_value9(acc1, e, sm.rexp[il] + sm.cexp[jl1] - 2056);
      res[0][e] = s0 == 0 ? y0 : res[0][e] + y0;
      res[1][e] = s0 == 0 ? y1 : res[1][e] + y1;
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = i0 + 16 * ti + g + 8 * (e >> 1), j = j0 + 8 * (tj0 + h) + 2 * t4 + (e & 1);
      if (i < Mr && j < Nc && (!sym || j >= i)) {
        double v = res[h][e];
        if (dsub && i == j) v -= (dsub[i] < 0) ? -1.0 : 1.0;
        C[(size_t)j * ldc + i] = v;
        if (sym && j > i) C[(size_t)i * ldc + j] = v;
      }
    }
}

size_t oz_gemm_smem_bytes() { return sizeof(OzGemmSmem); }

// Launch with the grid of k_gemm_oz; sets the kernel's shared-memory limit on first use per
// device (outside any stream capture: the solvers call it before capturing).
int oz_gemm_launch(int Mr, int Nc, int K, const double* A, int lda, int transA, const double* B, int ldb,
                   const int8_t* sb, const int8_t* dsub, double* C, int ldc, int sym, int transB, long long sa,
                   long long sbb, long long sc, int batch, cudaStream_t st) {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
      if (cudaFuncSetAttribute(k_gemm_oz, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OzGemmSmem)) !=
          cudaSuccess)
        return 1;
      done[dev] = true;
    }
  }
  const dim3 grid((Mr + OZM_TI - 1) / OZM_TI, (Nc + OZM_TJ - 1) / OZM_TJ, batch);
  k_gemm_oz<<<grid, 256, sizeof(OzGemmSmem), st>>>(Mr, Nc, K, A, lda, transA, B, ldb, sb, dsub, C, ldc, sym, transB,
                                                    sa, sbb, sc);
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace jac
