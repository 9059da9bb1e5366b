/* Internal declarations shared by the library's translation units. */
#ifndef OURO_INTERNAL_CUH
#define OURO_INTERNAL_CUH

#include <cuda_runtime.h>

#include "ouro.h"
#include "ouro_device.cuh"

/* Queue positions that kernels can hold at once on the GPU's 152 SMs: one per
 * resident thread (2048 an SM) in most kernels, four per thread in those of
 * large batches. */
#define OURO_SMS 152ull
#define OURO_BATCH_POS 4ull
/* Ring slack: consumers that hold one position per resident thread never make a
 * producer of a ring of (capacity + slack) slots wait one lap behind them.  The
 * batch malloc can hold 622,592 positions (1024 threads an SM); should they all
 * be of one class, beside a full queue of it, a producer waits for the oldest of
 * them, which does not wait for that producer.  More slack costs more than such
 * a wait: it doubles the rings of some heaps (12 GiB of 8 KiB pages: 2^22 slots
 * for 2^21, rounds of 965,676 mixed requests with one word each 121 -> 130 us). */
#define OURO_RING_SLACK (1ull << 19)
static_assert(OURO_RING_SLACK >= OURO_SMS * 2048, "ring slack below the resident threads");
/* Virtualized-array directories also span positions that are waiting for a
 * producer or in flight: four per thread, whatever kernel holds them. */
#define OURO_VA_SLACK (19ull << 16)
static_assert(OURO_VA_SLACK >= OURO_SMS * 2048 * OURO_BATCH_POS, "directory slack below the positions in flight");
/* work slots of fused rounds: one per stream that launches them on a heap (up
 * to this many), each on its own 128-byte line; zero between launches */
#define OURO_WORK_SLOTS 64

struct ouro_heap {
  ouro_heap_dev d;
  int device;
  void *heap_buf;
  int owns_heap;
  unsigned char *meta;          /* one device allocation for every metadata table */
  size_t meta_bytes;
  size_t off_qhdr, off_glob, off_stats, off_cls, off_pool, off_free, off_bits, off_cells, off_work;
  unsigned long long work_stream[OURO_WORK_SLOTS];   /* stream that slot k belongs to: its id + 1; 0: none (atomic) */
  size_t stats_words;
  unsigned long long ring_total;
  ouro_options opt;
};

namespace ouro {
namespace host {
extern thread_local int g_last_cuda_error;
ouro_status cuda_fail(cudaError_t e);
void count_launch(unsigned n = 1);
int sm_count();
/* ouro_round_fused, its arguments checked, with a given work slot (null: none) */
ouro_status round_fused_on(ouro_heap *H, const uint32_t *d_sizes, size_t n, uint32_t seed, int mode, ouro_check *d_out,
                           void **d_ptrs, void *work, cudaStream_t s);

/* Requests that a warp of the fused kernels takes at a time, 2^0 .. 2^5, for
 * n requests on `warps` resident warps.  A warp walks its larger blocks one
 * after another and every allocator step is a chain of L2 round trips, so up
 * to eight requests per warp go out as one task each (32 batches of 256 to
 * 8192 requests: 62 us a round with tasks of 32, 11 so).  Beyond that a warp
 * gets at least four tasks, so that the last ones fill the gaps, of at least
 * eight requests, which share their queue atomics.  Without a stage every
 * request goes to its queue, so there up to 16 requests share a task at once,
 * and 32 as soon as that leaves one and a half tasks per warp (page array,
 * tasks of 8 / 16 / 32: 110,000 sizes up to 4096 B 79 / 78 / 72 us, up to 8192
 * B 111 / 118 / 106, 262,144 of the size sweep 135 / 126 / 113, up to 8192 B 231
 * / 223 / 237; 200,000 up to 8192 B 185 / 180 / 210).  On chunk queues the steps
 * that a task's requests share (pop, reserve, claim, queue again) cost more
 * than uneven ends do, so their tasks go up to 32 requests first, with half
 * of the warps idle if need be (200,003 requests on the staged virtualized
 * array: tasks of 16 153 us, of 32 140; 30,011 on the chunk array: tasks of 16
 * 124 us, of 32 105; 3001: tasks of 4 56 us, of 32 80). */
inline unsigned round_task(unsigned long long n, unsigned long long warps, bool page_queues, bool staged) {
  const unsigned shared = !page_queues ? 32u : staged ? 8u : 16u, rounds = !page_queues || staged ? 8 : 3;
  unsigned t = 1;
  while (t < shared && t * warps < (page_queues ? n : 2 * n)) t *= 2;
  while (t < 32 && rounds * t * warps <= n) t *= 2;
  return t;
}
}  // namespace host
}  // namespace ouro

namespace ouro {
namespace host {
/* Launch with programmatic stream serialisation: the kernel's blocks may be
 * set up while the kernel before it on the stream still runs, and wait in
 * ouro::chain_begin() for it to finish.  Every kernel launched so calls
 * chain_begin() before it touches memory.  Between short kernels that set-up
 * is a good part of the time: four launches of 1024 requests 21.7 -> 16.8 us,
 * a fused round of 10,240 requests 12.4 -> 11.1, four launches of 2^20 mixed
 * requests with one word stored in each 109 -> 102.  Replayed graphs gained
 * nothing. */
template <typename... P, typename... A>
inline void launch_chained(void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);   /* errors: OURO_LAUNCHED */
}
}  // namespace host

/* Waits until the kernels before this one on the stream have finished and
 * their writes are visible, then lets the next chained kernel be set up: by
 * then this kernel's blocks are running, so it takes no place from them. */
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
}  // namespace ouro

#define OURO_CUDA(call)                                            \
  do {                                                             \
    cudaError_t e_ = (call);                                       \
    if (e_ != cudaSuccess) return ouro::host::cuda_fail(e_);       \
  } while (0)

#define OURO_LAUNCHED()                                            \
  do {                                                             \
    cudaError_t e_ = cudaGetLastError();                           \
    if (e_ != cudaSuccess) return ouro::host::cuda_fail(e_);       \
    ouro::host::count_launch();                                    \
  } while (0)

#endif
