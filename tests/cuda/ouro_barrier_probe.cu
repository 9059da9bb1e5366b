/* The grid barrier with blocks that never come (tests/test_gpu_barrier.py). */
#include "ouro_barrier.cuh"

__global__ void k_barrier_probe(unsigned long long *ctl, unsigned nblocks, unsigned limit, int *passed) {
  unsigned epoch = 0;
  const bool ok = ouro::detail::grid_barrier(ctl, nblocks, limit, epoch);
  if (threadIdx.x == 0) passed[blockIdx.x] = ok;
}

/* `blocks` blocks arrive at a barrier of nblocks and wait at most `limit` polls each */
extern "C" int barrier_probe(unsigned long long *ctl, unsigned nblocks, unsigned blocks, unsigned limit, int *passed) {
  k_barrier_probe<<<blocks, 64>>>(ctl, nblocks, limit, passed);
  return (int)cudaDeviceSynchronize();
}
