/*
 * Batching: many request batches of uneven size, each request allocating,
 * writing its pattern, reading it back and freeing (the driver round of
 * Sec. 3 of arXiv 2504.18211, applied to a stream of batches).
 *
 * Forms:
 *   - per launch:  one fused-round launch per batch (ouro_round_fused), or
 *                  four launches per batch (malloc / write / check / free);
 *   - CUDA graph:  the per-batch launches captured once and replayed;
 *   - persistent:  ONE kernel for all batches; warps pull tasks of 256
 *                  requests, and single rounds of 32 or fewer at the end of
 *                  a pass, from a device work counter, so uneven batches
 *                  overlap and the allocator state never leaves L2 between
 *                  them.
 * Request i of batch b uses pattern seed (seed + b) and thread id i (its
 * index inside the batch), in every form, so the per-batch checks agree.
 */
#include <algorithm>
#include <vector>

#include "ouro_internal.cuh"
#include "ouro_payload.cuh"
#include "ouro_shard.cuh"

using namespace ouro::detail;

namespace {

constexpr unsigned TASK_REQ_LOG = 8;   /* 256 requests per persistent task (the offsets' unit, see ouro.h) */

/* Warps claim work in rounds of 2^round_log requests: 32, or fewer on a pass
 * too short to give every resident warp a round of 32.  Round r of the launch
 * is round r mod R of task r / R, R = 256 >> round_log (a batch's last
 * task may have empty rounds).  A claim is a whole task until `last_wave`,
 * then one round: with whole tasks to the end a warp had 4 or 5 of them on a
 * pass of 6 M requests, and the kernel ended with the fives (96 batches of up
 * to 2^18 requests, staged: 3.22 ms, 3.05 so on one box; whole passes differ by
 * a tenth from box to box, 3.05 to 3.44 ms since). */
template <int V, bool STAGE>
__global__ void __launch_bounds__(256, ouro_page_queues(V) ? 4 : 2)   /* chunk queues: no spills at 2 per SM */
k_batches_persistent(ouro_heap_dev h, const uint32_t *sizes, const unsigned long long *offs,
                     const unsigned long long *task_offs, unsigned n_batches, uint32_t seed, int mode,
                     ouro_check *out, unsigned long long *work, unsigned long long n_rounds,
                     unsigned long long last_wave, unsigned round_log) {
  __shared__ ouro_block_ctx<8> ctx;
  if (STAGE) ouro_block_begin(ctx);
  const unsigned lane = laneid(), rpt_log = TASK_REQ_LOG - round_log;   /* rounds per task */
  payload_acc a;
  unsigned long long nulls = 0, next = 0, end = 0;
  unsigned b = 0;
  bool any = false;                        /* a holds counts of batch b */
  unsigned long long task_lo = 0, task_hi = 0, base = 0, count = 0;   /* tasks, requests of batch b */
  for (;;) {
    if (next == end) {
      const unsigned take = end < last_wave ? 1u << rpt_log : 1u;
      if (lane == 0) next = atomicAdd(work, (unsigned long long)take);
      next = __shfl_sync(0xffffffffu, next, 0);
      if (next >= n_rounds) break;
      end = next + take;
    }
    const unsigned long long task = next >> rpt_log;
    if (task < task_lo || task >= task_hi) {
      if (next >= n_rounds) break;
      if (any) warp_flush(a, nulls, &out[b]);
      a = payload_acc();
      nulls = 0;
      any = false;
      unsigned lo = 0, hi = n_batches;       /* task_offs[lo] <= task < task_offs[hi] */
      while (hi - lo > 1) {
        const unsigned mid = (lo + hi) >> 1;
        if (task_offs[mid] <= task) lo = mid;
        else hi = mid;
      }
      b = lo;
      task_lo = task_offs[b];
      task_hi = task_offs[b + 1];
      base = offs[b];
      count = offs[b + 1] - base;
    }
    const unsigned long long i = ((next - (task_lo << rpt_log)) << round_log) + lane;
    ++next;
    const bool active = lane >> round_log == 0 && i < count;
    if (!__any_sync(0xffffffffu, active)) continue;
    any = true;
    const uint32_t sz = active ? sizes[base + i] : 0;
    unsigned char *p = nullptr;
    if (STAGE) p = static_cast<unsigned char *>(stage_malloc_v<V>(ctx, h, sz, active));
    else p = static_cast<unsigned char *>(malloc_v<V>(h, sz, active));
    if (active && !p) nulls++;
    __syncwarp();
    warp_payload<PAY_FUSED, plain_payload(V, STAGE), pace_payload(V, STAGE)>(p, sz, (uint32_t)i, seed + b, mode, a,
                                                                             round_log >= 4);
    __syncwarp();
    if (STAGE) ouro::detail::stage_free<V, 8>(ctx, h, p, __activemask(), p ? size_class(h, sz) : -1);
    else free_v<V>(h, p);
    __syncwarp();
  }
  if (any) warp_flush(a, nulls, &out[b]);
  if (STAGE) ouro_block_end_v<V>(ctx, h);
}

#if OURO_SHARD_ENTRIES
inline cudaStream_t S(void *s) { return reinterpret_cast<cudaStream_t>(s); }
#endif

}  // namespace

/* ------------------------------------------------------- per-form launchers */
namespace ouro {
namespace launch {

template <int V, bool STAGE>
int persistent_blocks_per_sm(int blocks_per_sm) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batches_persistent<V, STAGE>, 256, 0);
  if (blocks_per_sm > 0 && blocks_per_sm < per_sm) per_sm = blocks_per_sm;
  return per_sm;
}

template <int V, bool STAGE>
ouro_status batches_form(ouro_heap *H, const uint32_t *d_sizes, const unsigned long long *d_offs,
                         const unsigned long long *d_task_offs, uint32_t n_batches, uint64_t n_tasks, uint32_t seed,
                         int mode, ouro_check *d_out, unsigned long long *d_work, int blocks_per_sm, cudaStream_t s) {
  const int grid = std::max(1, persistent_blocks_per_sm<V, STAGE>(blocks_per_sm)) * ouro::host::sm_count();
  const unsigned long long warps = 8ull * grid, requests = n_tasks << TASK_REQ_LOG;
  unsigned round_log = 0;
  for (unsigned t = ouro::host::round_task(requests, warps, ouro_page_queues(V), STAGE); t > 1; t >>= 1) ++round_log;
  /* single rounds for the last two tasks' worth per warp */
  const unsigned long long rounds = requests >> round_log, tail = (2 * warps) << (TASK_REQ_LOG - round_log);
  k_batches_persistent<V, STAGE><<<grid, 256, 0, s>>>(H->d, d_sizes, d_offs, d_task_offs, n_batches, seed, mode, d_out,
                                                      d_work, rounds, rounds > tail ? rounds - tail : 0, round_log);
  OURO_LAUNCHED();
  return OURO_OK;
}

template <int V>
ouro_status batches_persistent(ouro_heap *H, const uint32_t *d_sizes, const unsigned long long *d_offs,
                               const unsigned long long *d_task_offs, uint32_t n_batches, uint64_t n_tasks,
                               uint32_t seed, int mode, ouro_check *d_out, unsigned long long *d_work,
                               int blocks_per_sm, cudaStream_t s) {
  return H->d.staging ? batches_form<V, true>(H, d_sizes, d_offs, d_task_offs, n_batches, n_tasks, seed, mode, d_out,
                                              d_work, blocks_per_sm, s)
                      : batches_form<V, false>(H, d_sizes, d_offs, d_task_offs, n_batches, n_tasks, seed, mode, d_out,
                                               d_work, blocks_per_sm, s);
}

/* blocks of 256 per SM the unstaged persistent kernel keeps resident */
template <int V>
int batches_max_blocks_per_sm() { return persistent_blocks_per_sm<V, false>(0); }

#define INST_BATCHES_PERSISTENT(PRE, V)                                                                         \
  PRE template ouro_status batches_persistent<V>(ouro_heap *, const uint32_t *, const unsigned long long *,   \
                                                 const unsigned long long *, uint32_t, uint64_t, uint32_t, int, \
                                                 ouro_check *, unsigned long long *, int, cudaStream_t);
#define INST_BATCHES_MAX_BLOCKS(PRE, V) PRE template int batches_max_blocks_per_sm<V>();
OURO_SHARD_INSTANTIATE(INST_BATCHES_PERSISTENT)
OURO_SHARD_INSTANTIATE(INST_BATCHES_MAX_BLOCKS)

}  // namespace launch
}  // namespace ouro

#if OURO_SHARD_ENTRIES
struct ouro_batch_graph {
  cudaGraph_t graph;
  cudaGraphExec_t exec;
  size_t nodes;
  size_t kernels;   /* kernel nodes: the library's launches per replay */
  void *work;       /* its rounds' work slot; null: they work in their results (no memory for a slot) */
};

/* The graph's own work slot, zero: its rounds are one chain and a graph never
 * runs beside itself, so they share it.  Null where there is no memory for it.
 * Another thread may be capturing: nothing here touches its streams. */
static void *graph_work(cudaStream_t s) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  cudaThreadExchangeStreamCaptureMode(&mode);
  void *work = nullptr;
  if (cudaMalloc(&work, 128) != cudaSuccess) {
    cudaGetLastError();
    work = nullptr;
  } else if (cudaMemsetAsync(work, 0, 128, s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(work);
    work = nullptr;
  }
  cudaThreadExchangeStreamCaptureMode(&mode);
  return work;
}

/* waits for the replays in flight */
static void graph_work_free(void *work) {
  if (!work) return;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  cudaThreadExchangeStreamCaptureMode(&mode);
  cudaFree(work);
  cudaThreadExchangeStreamCaptureMode(&mode);
}

extern "C" ouro_status ouro_batches_persistent(ouro_heap *H, const uint32_t *d_sizes, const unsigned long long *d_offs,
                                               const unsigned long long *d_task_offs, uint32_t n_batches,
                                               uint64_t n_tasks, uint32_t seed, int mode, ouro_check *d_out,
                                               unsigned long long *d_work, int blocks_per_sm, void *stream) {
  if (!H || !d_sizes || !d_offs || !d_task_offs || !d_out || !d_work || n_batches == 0) return OURO_EINVAL;
  if (mode != 0 && mode != 1) return OURO_EINVAL;
  OURO_CUDA(cudaMemsetAsync(d_out, 0, sizeof(ouro_check) * n_batches, S(stream)));
  OURO_CUDA(cudaMemsetAsync(d_work, 0, 8, S(stream)));
  if (!n_tasks) return OURO_OK;
  OURO_DISPATCH(H->d.variant,
                return ouro::launch::batches_persistent<V>(H, d_sizes, d_offs, d_task_offs, n_batches, n_tasks, seed,
                                                           mode, d_out, d_work, blocks_per_sm, S(stream)));
}

extern "C" int ouro_batches_max_blocks_per_sm(const ouro_heap *H) {
  if (!H) return 0;
  switch (H->d.variant) {
#define CASE_MAX_BLOCKS(PRE, V) \
  case V: return ouro::launch::batches_max_blocks_per_sm<V>();
    OURO_SHARD_EACH(CASE_MAX_BLOCKS, )
#undef CASE_MAX_BLOCKS
    default: return 0;
  }
}

/* Capture the per-batch launches of one pass over all batches.
 * form 0: one fused-round launch per batch; form 1: malloc / write / check
 * / free per batch (d_ptrs: device scratch of max batch size pointers).
 * h_offs: HOST array of n_batches+1 request offsets into d_sizes. */
extern "C" ouro_status ouro_batch_graph_create(ouro_heap *H, const uint32_t *d_sizes, const unsigned long long *h_offs,
                                               uint32_t n_batches, uint32_t seed, int mode, ouro_check *d_out,
                                               void **d_ptrs, int form, ouro_batch_graph **out) {
  if (!H || !d_sizes || !h_offs || !d_out || !out || n_batches == 0 || (form == 1 && !d_ptrs) || form < 0 || form > 1)
    return OURO_EINVAL;
  if (mode != 0 && mode != 1) return OURO_EINVAL;
  *out = nullptr;
  cudaStream_t cs;
  OURO_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  ouro_status st = OURO_OK;
  cudaGraph_t g = nullptr;
  void *work = form == 0 ? graph_work(cs) : nullptr;
  cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) {
    graph_work_free(work);
    cudaStreamDestroy(cs);
    return ouro::host::cuda_fail(e);
  }
  for (uint32_t b = 0; b < n_batches && st == OURO_OK; ++b) {
    const size_t n = (size_t)(h_offs[b + 1] - h_offs[b]);
    const uint32_t *sz = d_sizes + h_offs[b];
    if (form == 0) {
      st = ouro::host::round_fused_on(H, sz, n, seed + b, mode, d_out + b, nullptr, work, cs);
    } else {
      st = ouro_batch_malloc(H, sz, d_ptrs, n, cs);
      if (st == OURO_OK) st = ouro_pattern_write(d_ptrs, sz, n, seed + b, mode, cs);
      if (st == OURO_OK) st = ouro_pattern_check(d_ptrs, sz, n, seed + b, mode, d_out + b, cs);
      if (st == OURO_OK) st = ouro_batch_free(H, d_ptrs, n, cs);
    }
  }
  e = cudaStreamEndCapture(cs, &g);
  if (st == OURO_OK && e != cudaSuccess) st = ouro::host::cuda_fail(e);
  ouro_batch_graph *G = nullptr;
  if (st == OURO_OK) {
    G = new ouro_batch_graph{g, nullptr, 0, 0, work};
    e = cudaGraphInstantiate(&G->exec, g, 0);
    if (e != cudaSuccess) st = ouro::host::cuda_fail(e);
    cudaGraphGetNodes(g, nullptr, &G->nodes);
    std::vector<cudaGraphNode_t> nodes(G->nodes);
    if (G->nodes) cudaGraphGetNodes(g, nodes.data(), &G->nodes);
    for (auto nd : nodes) {
      cudaGraphNodeType t;
      if (cudaGraphNodeGetType(nd, &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) G->kernels++;
    }
  }
  cudaStreamDestroy(cs);
  if (st != OURO_OK) {
    if (G) {
      if (G->exec) cudaGraphExecDestroy(G->exec);
      delete G;
    }
    if (g) cudaGraphDestroy(g);
    graph_work_free(work);
    return st;
  }
  *out = G;
  return OURO_OK;
}

extern "C" ouro_status ouro_batch_graph_launch(ouro_batch_graph *G, void *stream) {
  if (!G) return OURO_EINVAL;
  OURO_CUDA(cudaGraphLaunch(G->exec, S(stream)));
  ouro::host::count_launch((unsigned)G->kernels);
  return OURO_OK;
}

extern "C" uint64_t ouro_batch_graph_nodes(const ouro_batch_graph *G) { return G ? G->nodes : 0; }

extern "C" ouro_status ouro_batch_graph_destroy(ouro_batch_graph *G) {
  if (!G) return OURO_OK;
  cudaGraphExecDestroy(G->exec);
  cudaGraphDestroy(G->graph);
  graph_work_free(G->work);
  delete G;
  return OURO_OK;
}
#endif
