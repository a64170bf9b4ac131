// pair_cache.cuh -- skipping pairs whose outcome is already known, exactly.
//
// The Gram block A_P of a pair (Eq. (3.4)) depends only on the columns of its two blocks, and every
// step kernel is deterministic.  So when neither block has changed since the pair was last
// evaluated in the same slot of the same step, and it did not rotate then, its Gram block, the
// pivot's decision (no rotation) and its statistics would come out bitwise as before: the step
// kernels return at once for it, and the sweep reduction reads the statistics it left.  Late
// sweeps, where few pairs still rotate, then cost little more than the pairs that do.  Versions
// count the rotations that touched each block; a pair's record holds the versions it saw.
// Off for the per-cycle weight ordering (its slots change from sweep to sweep).
//
// The Gram kernel and the pivot look the pair up themselves; the pivot that decides it keeps the
// record (a block handed over to the FP64 pivot is recorded there; a failed one not at all).  The
// pairs of a step are disjoint, so no other CTA touches the versions of its two blocks in that step.
// (A kernel of its own between the steps cost 2.5 us per step, of the 55 to 85 us that a step of one
// problem of order 64 to 1501 takes.)
#pragma once
#include "jacobi_common.cuh"

namespace jac {

__device__ __forceinline__ bool pair_known(const JacProb& a, int s, int pair) {
  if (!a.pver) return false;
  const size_t i = (size_t)s * a.half + pair;
  const int4 e = a.pver[i];
  return e.x == a.pairs[2 * i] && e.y == a.pairs[2 * i + 1] && e.x >= 0 && e.z == a.bver[e.x] && e.w == a.bver[e.y];
}

// All threads of the pivot: a known pair is skipped by the update, and its statistics stay without the work.
__device__ __forceinline__ bool pair_skip_known(const JacProb& a, int s, int pair) {
  if (!pair_known(a, s, pair)) return false;
  if (threadIdx.x == 0) {
    a.skip[pair] = 1;
    PairStat& st = a.stats[(size_t)s * a.half + pair];
    st.inner_sweeps = 0;
    st.ns_steps = 0;
    st.evaluated = 0;
    for (int u = 0; u < 4; ++u) st.cyc[u] = 0;
  }
  return true;
}

// One thread, once the pair is decided.
__device__ __forceinline__ void pair_record(const JacProb& a, int s, int pair, bool rotated) {
  if (!a.pver) return;
  const size_t i = (size_t)s * a.half + pair;
  const int p = a.pairs[2 * i], q = a.pairs[2 * i + 1];
  const int vp = a.bver[p] + (rotated ? 1 : 0), vq = a.bver[q] + (rotated ? 1 : 0);
  if (rotated) {
    a.bver[p] = vp;
    a.bver[q] = vq;
  }
  a.pver[i] = make_int4(p, q, rotated ? -1 : vp, vq);
}

}  // namespace jac
