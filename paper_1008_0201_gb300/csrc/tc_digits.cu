// tc_digits.cu -- the FP64-accurate block update (Algorithm 3.4: [G_p G_q] <- [G_p G_q] V_P, and
// the same for V) from exact FP16 digit products on the fifth-generation tensor cores.
//
// Arithmetic and layout:
//   - a CTA takes 128-row tiles of Gw (then Vw) of one pair; per tile the columns are brought to
//     a common size (X~ = X D^-1, V~ = D V_P, D = diag(2^c_k), c_k the bound exponent of tile
//     column k), the rows of X~ and the columns of V~ are the scale groups, and every value
//     becomes 8 balanced 7-bit digits (ozaki.cuh), each an FP16 integer;
//   - the digits are written as K-major operands with the 128-byte swizzle (X~: 8 planes of
//     128 rows x 64 K; V~: 8 planes of 64 columns x 64 K) and one thread issues
//     tcgen05.mma kind::f16 (M = 128, K = 16, N = 64 per plane of V~, up to four planes at once)
//     for the digit pairs (t, u), t + u <= 8; products are exact and the level sums
//     acc_L = sum_{t+u=L} d_t d_u stay below 2^23 (64-term contraction), where the FP32 accumulation in
//     tensor memory is exact;
//   - levels 0..7 fill the 512 tensor-memory columns (one 64-column block per level); level 8
//     reuses block 0 once level 0 has been read;
//   - each thread reads its row's level sums for 16 output columns, gathers them exactly in two
//     int64 (levels 0..3 and 4..8) and rounds hi 2^35 + lo once to double in integer arithmetic
//     (oz_assemble.h): no FP64 instruction on the path.
// Grid (nx, 1, nprob), 512 threads, ~195 KB of shared memory (one CTA per SM): a persistent CTA
// walks the (pair, tile) items of its problem with stride nx; the items of pairs that did not
// rotate (skip flag of the pivot) cost one flag read.
#include <cooperative_groups.h>

#include "jacobi_common.cuh"
#include "pair_cache.cuh"
#include "oz_assemble.h"
#include "ozaki.cuh"
#include "tc.cuh"

namespace cg = cooperative_groups;

namespace jac {

namespace {
__device__ __forceinline__ unsigned char* align1k_d(unsigned char* p) {
  return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}
}  // namespace

#define TD_XPLANE 16384                       // 128 rows x 128 B
#define TD_VPLANE 8192                        // 64 rows x 128 B
#define TD_XOFF 0
#define TD_VOFF (OZ_T * TD_XPLANE)            // 131072
#define TD_MISC (TD_VOFF + OZ_T * TD_VPLANE)  // 196608: cexp[64], rexp[128], vexp[64], barriers
#define TD_SMEM (1024 + TD_MISC + 1024 + 128)
#define TD_NO_EXP (-100000)

size_t tc_update_oz_smem_bytes() { return TD_SMEM; }

__global__ void __launch_bounds__(512, 1) k_update_oz_tc(const JacProb* __restrict__ probs, int s) {
  extern __shared__ unsigned char td_raw[];
  unsigned char* sm = align1k_d(td_raw);
  int* cexp = reinterpret_cast<int*>(sm + TD_MISC);
  int* rexp = cexp + 64;
  int* vexp = rexp + 128;
  uint64_t* bar = reinterpret_cast<uint64_t*>(vexp + 64);  // [0] levels 0..7, [1] level 8
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
  const JacProb& a = probs[blockIdx.z];
  if (!a.active || s >= a.nsteps) return;
  const int gtiles = (a.mp + 127) >> 7;
  const int ntiles = gtiles + (a.Vw ? (a.np + 127) >> 7 : 0);
  const int nitems = a.counts[s] * ntiles;
  if ((int)blockIdx.x >= nitems) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    tc::mbar_init(&bar[0], 1);
    tc::mbar_init(&bar[1], 1);
    tc::fence_barrier_init();
  }
  if (warp == 0) tc::tmem_alloc(tslot, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tb = *tslot;
  const uint32_t xs = tc::smem_u32(sm + TD_XOFF), vs = tc::smem_u32(sm + TD_VOFF);
  // tile row r and output columns 16 cq .. + 15 of this thread, for the loads and digits of X~
  // and for the epilogue (warp w reads TMEM lanes 32 (w & 3) .. + 31: tid & 127 = r)
  const int r = tid & 127, cq = tid >> 7;
  const int vc = tid >> 3, vk0 = 8 * (tid & 7);  // V_P: column vc, rows (slab columns) vk0 .. + 7
  const uint32_t lrow = tb + ((uint32_t)(32 * (warp & 3)) << 16) + 16 * cq;
  bool bad = false;
  int it = 0;
  // The tile after the current one is loaded while the tensor cores work on the current one: the
  // lookups of a tile and its loads are one chain of dependent reads, 12 of 49 thousand clocks of a
  // tile; with the loads ahead 4 of 43 (4000 problems of orders 8..128 64.1 -> 62.6 ms).
  struct Tile {
    int item, pair, op, oq, wp, k, ld, rows;
    double* col0;  // row r of the tile in column 0
  } nx;
  double x[16];
  auto fetch = [&](int item) {  // the first item from here on whose pair rotated
    int pair = 0;
    for (; item < nitems; item += gridDim.x) {
      pair = item / ntiles;
      if (!a.skip[pair]) break;
    }
    nx.item = item;
    if (item >= nitems) return;
    const int t = item - pair * ntiles;
    const int* sp = a.pairs + (size_t)s * a.half * 2;
    const int p = sp[2 * pair], q = sp[2 * pair + 1];
    nx.pair = pair;
    nx.op = a.boff[p];
    nx.wp = a.boff[p + 1] - nx.op;
    nx.oq = a.boff[q];
    nx.k = nx.wp + a.boff[q + 1] - nx.oq;
    const bool isg = t < gtiles;
    nx.ld = isg ? a.mp : a.np;
    const int r0 = (isg ? t : t - gtiles) << 7;
    nx.rows = min(128, nx.ld - r0);
    nx.col0 = (isg ? a.Gw : a.Vw) + r0 + r;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int c = 16 * cq + j;
      x[j] = (c < nx.k && r < nx.rows) ? nx.col0[(size_t)(c < nx.wp ? nx.op + c : nx.oq + c - nx.wp) * nx.ld] : 0.0;
    }
  };
  fetch(blockIdx.x);
  while (nx.item < nitems) {
    const Tile cur = nx;
    const int k = cur.k, rows = cur.rows, wp = cur.wp, op = cur.op, oq = cur.oq;
    const double* Vp = a.vp + (size_t)cur.pair * a.apld * a.apld;
    // What lies past the tile's rows or the pair's columns is not formed: a warp whose 32 rows or 16
    // columns lie past them rests, and the contraction takes ceil(k / 16) steps of 16.  (Operand rows
    // left unwritten reach only their own, unread, rows or columns of the product.)  One pair of 64 rows
    // and 16 columns 25.6 -> 17.9 us, 4000 problems of orders 8..128 819 -> 756 us (549 with the MMAs and loads
    // below).
    const int k16 = (k + 15) >> 4;
    const bool works = 32 * (warp & 3) < rows && cq < k16;  // uniform per warp: its part of X~ and of Y
    const bool vworks = vc < 16 * k16 && vk0 < 16 * k16;    // its part of V~
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = (vc < k && vk0 + j < k) ? __ldg(Vp + (size_t)vc * a.apld + vk0 + j) : 0.0;
    if (tid < 64) cexp[tid] = 0;
    if (tid < 128) rexp[tid] = TD_NO_EXP;
    __syncthreads();
    // ---- column bounds c_k of the tile (a warp holds 32 rows of 16 columns)
    if (works) {
      int e = 0;  // lane j: of column j
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int ej = (int)__reduce_max_sync(0xffffffffu, (unsigned)oz_bexp(x[j]));
        if (lane == j) e = ej;
      }
      if (lane < 16 && e > 0) atomicMax(&cexp[16 * cq + lane], e);
    }
    __syncthreads();
    // ---- row groups of X~ and column groups of V~
    if (works) {
      int m = TD_NO_EXP;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int ex = oz_bexp(x[j]);
        if (ex != 0) m = max(m, ex - cexp[16 * cq + j]);
      }
      if (m != TD_NO_EXP) atomicMax(&rexp[r], m);
    }
    {
      int mv = TD_NO_EXP;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int ev = oz_bexp(v[j]), ck = cexp[vk0 + j];
        if (ev != 0 && ck != 0) mv = max(mv, ev + ck);
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) mv = max(mv, __shfl_xor_sync(0xffffffffu, mv, o));
      if ((tid & 7) == 0) vexp[vc] = mv;
    }
    // the previous tile's MMAs were waited for before its epilogue: the planes are free
    __syncthreads();
    // ---- digits of X~ (row r) and of V~ (operand row vc): 16-byte stores, 8 K entries each
    if (works) {
      const int ea = rexp[r];
#pragma unroll
      for (int j0 = 0; j0 < 16; j0 += 8) {
        unsigned w[OZ_T][4];
#pragma unroll
        for (int jj = 0; jj < 8; jj += 2) {
          unsigned d[OZ_T];
          const int c0 = 16 * cq + j0 + jj;
          oz_split2(oz_biased(x[j0 + jj], oz_bexp(x[j0 + jj]) - cexp[c0] - ea),
                    oz_biased(x[j0 + jj + 1], oz_bexp(x[j0 + jj + 1]) - cexp[c0 + 1] - ea), d);
#pragma unroll
          for (int tt = 0; tt < OZ_T; ++tt) w[tt][jj >> 1] = d[tt];
        }
        const uint32_t off = tc::sw128_offset(r, 16 * cq + j0, 2);
#pragma unroll
        for (int tt = 0; tt < OZ_T; ++tt)
          *reinterpret_cast<uint4*>(sm + TD_XOFF + tt * TD_XPLANE + off) = make_uint4(w[tt][0], w[tt][1], w[tt][2],
                                                                                      w[tt][3]);
      }
    }
    if (vworks) {
      const int ev = vexp[vc];
      unsigned w[OZ_T][4];
#pragma unroll
      for (int jj = 0; jj < 8; jj += 2) {
        unsigned d[OZ_T];
        const int ck0 = cexp[vk0 + jj], ck1 = cexp[vk0 + jj + 1];
        oz_split2((ck0 != 0 && ev != TD_NO_EXP) ? oz_biased(v[jj], oz_bexp(v[jj]) + ck0 - ev) : OZ_BIAS,
                  (ck1 != 0 && ev != TD_NO_EXP) ? oz_biased(v[jj + 1], oz_bexp(v[jj + 1]) + ck1 - ev) : OZ_BIAS, d);
#pragma unroll
        for (int tt = 0; tt < OZ_T; ++tt) w[tt][jj >> 1] = d[tt];
      }
      const uint32_t off = tc::sw128_offset(vc, vk0, 2);
#pragma unroll
      for (int tt = 0; tt < OZ_T; ++tt)
        *reinterpret_cast<uint4*>(sm + TD_VOFF + tt * TD_VPLANE + off) = make_uint4(w[tt][0], w[tt][1], w[tt][2],
                                                                                    w[tt][3]);
    }
    tc::fence_proxy_async_smem();
    __syncthreads();
    // ---- levels 0..7: block L (TMEM columns 64 L ..) accumulates sum_{t+u=L} X_t V_u.  The planes of
    // V~ lie one after the other, so one MMA of N = 64 nb takes X_t against planes u .. u + nb - 1 into
    // blocks t + u .. t + u + nb - 1: 12 MMAs per 16 K in place of 36, each plane of X~ read once or
    // twice and no descriptor formed in the loop: 15.3 -> 5.3 thousand clocks of a full tile, which takes 43.
    const uint64_t dx = tc::desc_sw128(xs, 16, 1024), dv = tc::desc_sw128(vs, 16, 1024);
    if (tid == 0) {
      tc::fence_after_sync();
#pragma unroll 1
      for (int kk = 0; kk < k16; ++kk)
#pragma unroll
        for (int tt = 0; tt < OZ_T; ++tt)
#pragma unroll
          for (int u = 0; u < OZ_T - tt; u += 4) {
            const int nb = (OZ_T - tt - u < 4) ? OZ_T - tt - u : 4;
            tc::mma_f16(tb + 64 * (tt + u), dx + ((tt * TD_XPLANE + kk * 32) >> 4),
                        dv + ((u * TD_VPLANE + kk * 32) >> 4), tc::idesc_f32acc(tc::FMT_F16, 128, 64 * nb, 0, 0),
                        (kk > 0 || tt > 0) ? 1u : 0u);
          }
      tc::mma_commit(&bar[0]);
    }
    fetch(cur.item + gridDim.x);
    if (__syncthreads_or(!tc::mbar_wait(&bar[0], it & 1))) {
      bad = true;
      break;
    }
    tc::fence_after_sync();
    int q01[16];
    if (works) {
      uint32_t la[16], lb[16];
      tc::tmem_ld16(lrow, la);
      tc::tmem_ld16(lrow + 64, lb);
      tc::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 16; ++j)
        q01[j] = f32_small_int(__uint_as_float(la[j])) * 128 + f32_small_int(__uint_as_float(lb[j]));
    }
    tc::fence_before_sync();
    __syncthreads();  // level 0 read everywhere: block 0 is free for level 8
    if (tid == 0) {
      tc::fence_after_sync();
#pragma unroll 1
      for (int kk = 0; kk < k16; ++kk)
#pragma unroll
        for (int tt = 1; tt < OZ_T; ++tt)
          tc::mma_f16(tb, dx + ((tt * TD_XPLANE + kk * 32) >> 4), dv + (((8 - tt) * TD_VPLANE + kk * 32) >> 4),
                      tc::idesc_f32acc(tc::FMT_F16, 128, 64, 0, 0), (kk > 0 || tt > 1) ? 1u : 0u);
      tc::mma_commit(&bar[1]);
    }
    // four output columns at a time (more need all the registers and spill): levels 2..7, two levels
    // joined in 32 bits, then level 8
    const int ea = rexp[r];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      int q23[4], q45[4], q67[4];
      if (works) {
        uint32_t l[6][4];
#pragma unroll
        for (int u = 0; u < 6; ++u) tc::tmem_ld4(lrow + 64 * (u + 2) + 4 * h, l[u]);
        tc::tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          q23[j] = f32_small_int(__uint_as_float(l[0][j])) * 128 + f32_small_int(__uint_as_float(l[1][j]));
          q45[j] = f32_small_int(__uint_as_float(l[2][j])) * 128 + f32_small_int(__uint_as_float(l[3][j]));
          q67[j] = f32_small_int(__uint_as_float(l[4][j])) * 128 + f32_small_int(__uint_as_float(l[5][j]));
        }
      }
      if (h == 0) {
        if (__syncthreads_or(!tc::mbar_wait(&bar[1], it & 1))) {
          bad = true;
          break;
        }
        tc::fence_after_sync();
      }
      if (works) {
        uint32_t l8[4];
        tc::tmem_ld4(lrow + 4 * h, l8);
        tc::tmem_wait_ld();
        if (r < rows) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int c = 16 * cq + 4 * h + j;
            if (c < k) {
              const long long hi = (long long)q01[4 * h + j] * 16384 + q23[j];
              const long long lo = ((long long)q45[j] * 16384 + q67[j]) * 128 + f32_small_int(__uint_as_float(l8[j]));
              cur.col0[(size_t)(c < wp ? op + c : oq + c - wp) * cur.ld] =
                  oz_assemble_small(hi, lo, 35, ea + vexp[c] - 2056 - 56);
            }
          }
        }
      }
    }
    if (bad) break;
    tc::fence_before_sync();
    __syncthreads();  // TMEM and the exponent arrays read before the next tile reuses them
    ++it;
  }
  if (bad && tid == 0) {
    atomicOr(a.pflags, JAC_DEVERR_TIMEOUT);
    tc::mbar_wait(&bar[0], it & 1);
    tc::mbar_wait(&bar[1], it & 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tb, 512);
}

// ------------------------------------------------------------------------------------ Gram
// FP64-accurate Gram block A_P = X^T X (Eq. (3.4)) from exact FP16 digit products: grid
// (half * CS / VR, nprob), cluster (CS / VR, 1, 1), 512 threads: the rows of a pair fall into CS shares as
// in k_gram_oz, VR consecutive shares (1 or 2) to a CTA, with the same stages of 128 rows, scale groups
// (every column, bound exponent E_c), 8 digits, levels 0..7 and order of the FP64 additions: the two
// kernels give the same bits.
//
// tcgen05 layout.  The operand is X^T: 64 rows (the pair's columns) by 128 K (the stage's rows), as two
// 64-K chunks; inside a chunk the 8 digit planes follow each other (plane t at t * 8 KB).  So one
// M = 128 operand covers planes a and a + 1, and one N = 64 nb operand planes v .. v + nb - 1: an MMA puts
// D_a D_u^T (level a + u) in TMEM lanes 0..63 and D_{a+1} D_u^T (level a + u + 1) in lanes 64..127 of the
// 64-column block a + u, u = v .. v + nb - 1.  With a = 0, 2, 4, 6 and u <= 7 - a every product with
// t + u <= 7 is there once, in 6 MMAs per 16 K (20 with N = 64; 36 products); what reaches level 8
// lands in the lower lanes of block 7 and is not read.  Level L is the upper lanes of block L plus the
// lower lanes of block L - 1: each half gathers its share of a 16-column strip in integers, finishes 8
// of the columns and passes its share of the other 8 to the other half through shared memory.
// A_P is exactly symmetric (the level sums of (i, j) and (j, i) are the same integers), so only
// entries j >= i are formed.
// The MMAs take 4 thousand clocks of the 19 of a stage, where mma.sync (k_gram_oz) takes about half of
// 34; the digits take 5, the integer sums and their rounding 8.  32 pairs of 2304 rows: 94 us with
// k_gram_oz, 86 with one share per CTA, 67 with two; where it is the slower one: gram_tc_shares (capi.cu).
#define TGD_CHUNK 65536                        // 8 planes x 64 rows x 128 B
#define TGD_TOT (2 * TGD_CHUNK)                // FP64 partials [VR][64][65] after the digits
#define TGD_MISC (TGD_TOT + 2 * 64 * 65 * 8)
#define TGD_SMEM (1024 + TGD_MISC + 512 + 128)

size_t tc_gram_oz_smem_bytes() { return TGD_SMEM; }

__global__ void __launch_bounds__(512, 1) k_gram_oz_tc(const JacProb* __restrict__ probs, int s, int CS, int VR) {
  extern __shared__ unsigned char tgd_raw[];
  unsigned char* sm = align1k_d(tgd_raw);
  double* C = reinterpret_cast<double*>(sm + TGD_TOT);  // [VR][64][65], entries j >= i
  int* E = reinterpret_cast<int*>(sm + TGD_MISC);       // [64]
  uint64_t* bar = reinterpret_cast<uint64_t*>(E + 64);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 1);
  longlong2* xch = reinterpret_cast<longlong2*>(sm);    // [column][row], over the digits
  cg::cluster_group cluster = cg::this_cluster();
  const JacProb& a = probs[blockIdx.y];
  const int nc = CS / VR, pair = blockIdx.x / nc;
  const int crank = (int)cluster.block_rank();
  if (!a.active || s >= a.nsteps || pair >= a.counts[s]) return;
  const int* sp = a.pairs + (size_t)s * a.half * 2;
  const int p = sp[2 * pair], q = sp[2 * pair + 1];
  if (pair_known(a, s, pair)) return;  // uniform
  const int op = a.boff[p], wp = a.boff[p + 1] - op, oq = a.boff[q], wq = a.boff[q + 1] - oq;
  const int k = wp + wq;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rpc = ((a.mp / CS + 15) & ~15);
  auto begin_of = [&](int vr) { return min(a.mp, (crank * VR + vr) * rpc); };
  // warp w: columns 4 w .. 4 w + 3; lane l: stage rows 4 l .. 4 l + 3 (K-adjacent digits)
  double x[4][4];
  auto fetch = [&](int g0, int rs) {
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) {
      const int c = 4 * warp + cc;
      const double* col = a.Gw + (size_t)(c < wp ? op + c : oq + c - wp) * a.mp + g0;
#pragma unroll
      for (int i = 0; i < 4; i += 2) {
        const int rr = 4 * lane + i;
        const double2 v = (c < k && rr < rs) ? __ldg(reinterpret_cast<const double2*>(col + rr)) : make_double2(0.0, 0.0);
        x[cc][i] = v.x;
        x[cc][i + 1] = v.y;
      }
    }
  };
  fetch(begin_of(0), begin_of(1) - begin_of(0));
  if (tid == 0) {
    tc::mbar_init(&bar[0], 1);
    tc::fence_barrier_init();
  }
  if (warp == 0) tc::tmem_alloc(tslot, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tb = *tslot;
  const uint64_t dd = tc::desc_sw128(tc::smem_u32(sm), 16, 1024);
  // epilogue: warp w reads TMEM lanes 32 (w & 3) .. + 31 (operand rows) and the strip of columns
  // c0 = 16 (w >> 2) .. + 15; it finishes columns c0 .. + 7 (upper lanes) or c0 + 8 .. + 15
  const bool upper = (warp & 3) < 2;
  const int i = (32 * (warp & 3) + lane) & 63, c0 = 16 * (warp >> 2);
  const bool works = c0 + 15 >= (i & 32) && c0 < k && (i & 32) < k;  // uniform: some entry j >= i of the block
  const uint32_t laddr = tb + ((uint32_t)(32 * (warp & 3)) << 16) + c0;
  const int cf = c0 + (upper ? 0 : 8), cs = c0 + (upper ? 8 : 0);
  // this lane's share of eight columns from c (c0 or c0 + 8)
  auto gather = [&](int c, long long(&hi)[8], long long(&lo)[8]) {
    uint32_t lv[4][8];
    int qa[8], qb[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int L = 4 * h + u, B = L - (upper ? 0 : 1);  // uniform
        if (B >= 0) {
          tc::tmem_ld8(laddr + (c - c0) + 64 * B, lv[u]);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) lv[u][j] = 0;
        }
      }
      tc::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        qa[j] = f32_small_int(__uint_as_float(lv[0][j])) * 128 + f32_small_int(__uint_as_float(lv[1][j]));
        qb[j] = f32_small_int(__uint_as_float(lv[2][j])) * 128 + f32_small_int(__uint_as_float(lv[3][j]));
        (h ? lo[j] : hi[j]) = (long long)qa[j] * 16384 + qb[j];
      }
    }
  };
  double* out = a.Ap + (size_t)pair * a.apld * a.apld;
  bool bad = false;
  int it = 0;
  for (int vr = 0; vr < VR && !bad; ++vr) {
    const int r_begin = begin_of(vr), r_end = begin_of(vr + 1);
    double tot[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) tot[j] = 0.0;
    for (int g0 = r_begin; g0 < r_end; g0 += 128, ++it) {
      const int steps = (min(128, r_end - g0) + 15) >> 4;  // of 16 K
      int ec[4];
#pragma unroll
      for (int cc = 0; cc < 4; ++cc)
        ec[cc] = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(max(oz_bexp(x[cc][0]), oz_bexp(x[cc][1])),
                                                                   max(oz_bexp(x[cc][2]), oz_bexp(x[cc][3]))));
      if (lane == 0) *reinterpret_cast<int4*>(&E[4 * warp]) = make_int4(ec[0], ec[1], ec[2], ec[3]);
      // digits: operand row c (pair column), K = stage rows 4 lane .. + 3 (chunk lane >> 4)
      if (16 * steps > 4 * lane) {
        unsigned char* base = sm + (lane >> 4) * TGD_CHUNK;
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          unsigned long long b[4];
          unsigned w0[OZ_T], w1[OZ_T];
#pragma unroll
          for (int u = 0; u < 4; ++u) b[u] = oz_biased(x[cc][u], oz_bexp(x[cc][u]) - ec[cc]);
          oz_split2(b[0], b[1], w0);
          oz_split2(b[2], b[3], w1);
          const uint32_t off = tc::sw128_offset(4 * warp + cc, (4 * lane) & 63, 2);
#pragma unroll
          for (int tt = 0; tt < OZ_T; ++tt)
            *reinterpret_cast<uint2*>(base + tt * 8192 + off) = make_uint2(w0[tt], w1[tt]);
        }
      }
      tc::fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0) {
        tc::fence_after_sync();
#pragma unroll 1
        for (int kk = 0; kk < steps; ++kk) {
          const uint64_t dk = dd + (((kk >> 2) * TGD_CHUNK + (kk & 3) * 32) >> 4);
#pragma unroll
          for (int a0 = 0; a0 < OZ_T; a0 += 2)
#pragma unroll
            for (int v = 0; v < OZ_T - a0; v += 4) {
              const int nb = (OZ_T - a0 - v < 4) ? OZ_T - a0 - v : 4;
              tc::mma_f16(tb + 64 * (a0 + v), dk + ((a0 * 8192) >> 4), dk + ((v * 8192) >> 4),
                          tc::idesc_f32acc(tc::FMT_F16, 128, 64 * nb, 0, 0), (kk > 0 || a0 > 0) ? 1u : 0u);
            }
        }
        tc::mma_commit(&bar[0]);
      }
      if (g0 + 128 < r_end) fetch(g0 + 128, r_end - g0 - 128);
      else if (vr + 1 < VR) fetch(r_end, begin_of(vr + 2) - r_end);
      if (__syncthreads_or(!tc::mbar_wait(&bar[0], it & 1))) {
        bad = true;
        break;
      }
      tc::fence_after_sync();
      long long hi[8], lo[8];
      if (works) {
        gather(cs, hi, lo);
#pragma unroll
        for (int j = 0; j < 8; ++j) xch[(cs + j) * 64 + i] = make_longlong2(hi[j], lo[j]);
        gather(cf, hi, lo);
      }
      __syncthreads();
      if (works) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = cf + j;
          if (c >= i && c < k) {
            const longlong2 o = xch[c * 64 + i];
            const double y = oz_assemble_small(hi[j] + o.x, lo[j] + o.y, 28, E[i] + E[c] - 2056 - 49);
            tot[j] = (g0 == r_begin) ? y : tot[j] + y;
          }
        }
      }
      tc::fence_before_sync();
      __syncthreads();  // TMEM, the exchange and E read before the next stage overwrites them
    }
    if (works) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = cf + j;
        if (c < i || c >= k) continue;
        if (CS > 1) {
          C[vr * 64 * 65 + i * 65 + c] = tot[j];
        } else {  // nothing to add up
          out[c * a.apld + i] = tot[j];
          out[i * a.apld + c] = tot[j];
        }
      }
    }
  }
  if (bad && tid == 0) {
    atomicOr(a.pflags, JAC_DEVERR_TIMEOUT);
    tc::mbar_wait(&bar[0], it & 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tb, 512);
  if (CS == 1) return;
  cluster.sync();
  // the upper triangle, rows n and k - 1 - n together as one row of k + 1 entries (as k_gram_oz)
  const int totn = ((k + 1) >> 1) * (k + 1), per = (totn + nc - 1) / nc;
  const int e0 = crank * per, e1 = min(totn, e0 + per);
  for (int e = e0 + tid; e < e1; e += 512) {
    const int n = e / (k + 1), o = e - n * (k + 1);
    int ri = n, rj = n + o;
    if (rj >= k) {
      ri = k - 1 - n;
      rj = ri + (o - (k - n));
      if (ri == n) continue;  // the middle row of an odd block
    }
    double part[16];  // all remote loads issued before the fixed-order sum
#pragma unroll
    for (int rk = 0; rk < 16; ++rk)
      part[rk] = (rk < CS) ? cluster.map_shared_rank(C, rk / VR)[rk % VR * 64 * 65 + ri * 65 + rj] : 0.0;
    double sum = part[0];
#pragma unroll
    for (int rk = 1; rk < 16; ++rk)
      if (rk < CS) sum += part[rk];
    out[rj * a.apld + ri] = sum;
    out[ri * a.apld + rj] = sum;
  }
  cluster.sync();  // keep every partial alive until all remote reads are done
}

}  // namespace jac
