// pair_cache.cu -- set-up of the pair cache (pair_cache.cuh).
#include "jacobi_common.cuh"

namespace jac {

// Grid (nprob), 256 threads: no record valid, versions 0.
__global__ void k_cache_init(const JacProb* __restrict__ probs) {
  const JacProb& a = probs[blockIdx.x];
  if (!a.pver) return;
  for (int i = threadIdx.x; i < a.nsteps * a.half; i += blockDim.x) a.pver[i] = make_int4(-1, -1, -1, -1);
  for (int i = threadIdx.x; i < a.nb; i += blockDim.x) a.bver[i] = 0;
}

}  // namespace jac
