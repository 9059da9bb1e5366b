/* Grid barrier of the library's cooperative kernels. */
#ifndef OURO_BARRIER_CUH
#define OURO_BARRIER_CUH

#include "ouro_internal.cuh"

namespace ouro {
namespace detail {

/* ctl[0] counts arrivals and is never reset, the e-th barrier waits until it
 * reaches e * nblocks, so an arrival is one fence and one atomic, and the wait
 * polls that same word.  A wait that runs out sets ctl[4] and the count's
 * BARRIER_FAILED bit, which ends every other block's wait and the barrier of
 * every block that comes later.  The bit is or-ed in: the blocks that wait
 * give up together, and added by each it would carry out of the word. */
constexpr unsigned long long BARRIER_FAILED = 1ull << 62;

__device__ inline bool grid_barrier(unsigned long long *ctl, unsigned nblocks, unsigned limit, unsigned &epoch) {
  __shared__ int ok;
  __syncthreads();
  ++epoch;
  if (threadIdx.x == 0) {
    const unsigned long long target = (unsigned long long)nblocks * epoch;
    __threadfence();
    unsigned long long seen = atomicAdd(&ctl[0], 1ull) + 1;
    if (seen >= target) __threadfence();
    for (unsigned it = 0; seen < target; seen = ld_acq(&ctl[0])) {
      if (++it > limit) {
        atomicExch(&ctl[4], 1ull);
        atomicOr(&ctl[0], BARRIER_FAILED);
        seen = BARRIER_FAILED;
        break;
      }
      __nanosleep(32);
    }
    ok = seen < BARRIER_FAILED;
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace detail
}  // namespace ouro

#endif
