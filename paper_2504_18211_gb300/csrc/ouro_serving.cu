/*
 * Serving: a request loop that stays on the device (one cooperative,
 * persistent kernel for all steps) over sessions whose memory grows.
 *
 * Each step has two phases, with a grid barrier after each:
 *   1. growth (all blocks): every active session allocates one block with
 *      ouro_malloc, records it in its block table, writes its pattern (seed +
 *      session id, block index) and reads it back through L2, folding the
 *      words into the session checksum; a session that has reached its size
 *      reports its checksum, gives its slot back and is listed;
 *   2. freeing and admission: the listed sessions' blocks are cut into tasks
 *      of 32 (one round of a warp) dealt to the warps in turn, so that the
 *      step's frees spread over the grid and one long session does not hold
 *      the step for a single warp.  Meanwhile the grid's last warp admits the
 *      sessions of the next step, in arrival order, while a session slot is
 *      free and the blocks committed to admitted sessions, plus the
 *      newcomer's total, stay within the admission cap (95 % of the heap's
 *      blocks); it weighs 32 arrivals at a time and admits the longest run of
 *      them, from the first, that passes.  Admission needs slots and
 *      committed blocks, which phase 1 settled, and nothing that is freed.
 * The allocator state, the session table and the block tables stay resident
 * for the whole run; requests that arrive while others are running are
 * admitted as slots and memory free up, and their work overlaps on the GPU.
 * Step boundaries are a grid barrier of this file (every wait bounded); one
 * thread stamps %globaltimer after each step for the latency histogram.
 *
 * The same phases also run as the plain per-launch form (ouro_serve_per_launch):
 * one kernel per phase and step in stream order, kernel boundaries in place
 * of the grid barriers, for comparison with the one-launch loop.
 */
#include <algorithm>

#include "ouro_barrier.cuh"
#include "ouro_internal.cuh"
#include "ouro_payload.cuh"
#include "ouro_shard.cuh"

using namespace ouro::detail;

namespace {

struct serve_args {
  ouro_heap_dev h;
  /* sessions, in arrival order */
  const uint32_t *arrive_step;   /* step at which the session has arrived */
  const uint32_t *blocks;        /* total blocks the session grows to */
  uint32_t n_sessions;
  /* slots */
  uint32_t n_slots, max_blocks;
  int *slot_session;             /* session id, -1 free, -2 - id: admitted, no block yet */
  uint32_t *slot_k;              /* blocks allocated so far */
  unsigned long long *slot_acc;  /* per slot: xor, sum, mismatches */
  unsigned long long *tables;    /* n_slots x max_blocks block pointers */
  /* results */
  unsigned long long *sess_out;  /* per session: xor, sum, mismatches, admit step, done step (u64 each) */
  unsigned long long *step_ns;   /* per step: %globaltimer when its growth begins, when that has ended, and
                                    when its frees and the next admission have (3 words) */
  unsigned long long *ctl;       /* [0] barrier arrivals, [1] reserved, [2] next arrival,
                                    [3] committed blocks, [4] error, [5] mallocs, [6] frees, [7] failed,
                                    [8] free-slot stack top, [9 + step % 2] sessions finished this step */
  uint32_t *free_stack;          /* free slot ids (stack of n_slots) */
  uint32_t *done_list;           /* slots whose sessions finished this step (n_slots) */
  uint32_t steps;
  uint32_t seed;
  unsigned long long cap_blocks; /* admission cap */
  uint32_t block_bytes;
  uint32_t spin_limit;
};

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

/* ---------------------------------------------------------------- phases
 * Each phase is a device function over the whole grid; the cooperative
 * kernel separates them with grid barriers, the per-launch form with kernel
 * boundaries on one stream. */

/* the free-slot stack holds every slot */
__device__ void serve_init(const serve_args &A) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n_slots; i += gridDim.x * blockDim.x)
    A.free_stack[i] = A.n_slots - 1 - i;
  if (blockIdx.x == 0 && threadIdx.x == 0) A.ctl[8] = A.n_slots;
}

/* Admission for step `step` (the grid's last warp, the last to get freeing
 * tasks): arrival order, a free slot (stack), committed + newcomer <= cap.
 * Also empties the finished count that the step will use. */
__device__ void serve_admit(const serve_args &A, uint32_t step) {
  if (blockIdx.x != gridDim.x - 1 || threadIdx.x < blockDim.x - 32) return;
  const unsigned lane = laneid();
  if (lane == 0) A.ctl[9 + (step & 1)] = 0;
  unsigned long long next = A.ctl[2], committed = *(volatile unsigned long long *)&A.ctl[3],
                     top = *(volatile unsigned long long *)&A.ctl[8];
  for (;;) {
    const unsigned long long i = next + lane;
    const bool arrived = i < A.n_sessions && A.arrive_step[i] <= step;
    unsigned long long cum = arrived ? A.blocks[i] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, cum, o);
      if ((int)lane >= o) cum += y;
    }
    const bool ok = arrived && committed + cum <= A.cap_blocks && lane < top;
    const unsigned okm = __ballot_sync(0xffffffffu, ok);
    const unsigned n_adm = okm == 0xffffffffu ? 32u : (unsigned)(__ffs(~okm) - 1);   /* leading run */
    if (lane < n_adm) {
      const uint32_t slot = __ldcg(&A.free_stack[top - 1 - lane]);
      A.slot_session[slot] = -2 - (int)i;
      A.sess_out[5 * i + 3] = step;
    }
    if (n_adm) committed += __shfl_sync(0xffffffffu, cum, n_adm - 1);
    next += n_adm;
    top -= n_adm;
    if (n_adm < 32) break;
  }
  if (lane == 0) {
    A.ctl[2] = next;
    A.ctl[3] = committed;
    A.ctl[8] = top;
  }
  __threadfence();
}

/* Growth and completion.  Block b of the grid holds slots b, b + grid, ...,
 * up to 32 of them at a time: its first warp reads their sessions, a lane
 * each, and allocates all their blocks with one queue operation; then the
 * block's warps write the new blocks in pieces of SERVE_PIECE units, all of
 * them, and read them back, each warp what its neighbour wrote, eight loads
 * in flight per lane.  One warp per session had walked the allocator's chain
 * and 16 KiB alone, sessions one after another.  What is left is a chain of
 * L2 round trips, not bandwidth: 400 steps of about 1700 blocks of 16 KiB took
 * 12.3 ms with five barriers and phases a step, 8.0 ms so, 6.9 ms with the
 * sessions kept and grid_barrier on one word (28 MB a step would take 4.2 us of its
 * 17 at the copy rate). */
constexpr uint32_t SERVE_PIECE = 256;

/* One block of class cls for every lane with `want` (all 32 lanes call).  On
 * chunk queues the warp pops a chunk per lane at once, as the batch malloc
 * does: one class group of chunk_malloc pops them one after another, and a
 * serving block takes a chunk of its own where chunks are no larger (400 steps
 * of about 1700 blocks: chunk array 15.7 ms, 9.3 so, virtualized list 20.2 and
 * 12.3). */
template <int V>
__device__ __forceinline__ unsigned char *serve_malloc(const ouro_heap_dev &h, uint32_t bytes, bool want) {
  if constexpr (!ouro_page_queues(V)) {
    if (!h.deopt) {
      __shared__ unsigned items[32];
      const unsigned wm = __ballot_sync(0xffffffffu, want), need = __popc(wm), rank = __popc(wm & lanemask_lt());
      if (!need) return nullptr;
      const int cls = size_class(h, bytes);
      const unsigned got = chunk_acquire<V>(h, cls, need, items);
      __syncwarp();
      const unsigned item = want && rank < got ? items[rank] : OURO_NIL;
      const unsigned n = __popc(__ballot_sync(0xffffffffu, item != OURO_NIL));
      if (laneid() == 0) {
        stat_add(h, cls, OURO_ST_MALLOC, n);
        stat_add(h, cls, OURO_ST_FAILED, need - n);
      }
      return item != OURO_NIL ? h.base + ((size_t)item << (4 + cls)) : nullptr;
    }
  }
  /* (a step's growth can carve thousands of chunks: eight slot writes per
   *  lane in flight while the warp fills them) */
  return static_cast<unsigned char *>(malloc_v<V, 8>(h, bytes, want));
}

/* a lane's session between two steps of one launch */
struct serve_lane {
  unsigned long long x, sum, mism;
  int sess;                /* -1: none */
  uint32_t k, total;
};

/* keep (shared memory, one entry per lane of the first warp; null in the
 * per-launch form): the block's sessions stay there from step to step, for
 * grids that hold every slot at once, instead of being read back from memory
 * (two dependent L2 round trips a step).  k_serve writes those that are still
 * growing back when it ends. */
template <int V>
__device__ void serve_grow(const serve_args &A, uint32_t step, serve_lane *keep) {
  __shared__ unsigned char *s_bp[32];
  __shared__ uint32_t s_key[32];
  __shared__ unsigned long long s_sum[32];
  __shared__ unsigned s_xor[32], s_mism[32];
  __shared__ unsigned s_n;
  const unsigned lane = laneid(), warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const ouro_heap_dev &h = A.h;
  const uint32_t units = A.block_bytes >> 4, per = (units + SERVE_PIECE - 1) / SERVE_PIECE;
  for (unsigned long long first = blockIdx.x; first < A.n_slots; first += 32ull * gridDim.x) {
    int sess = -1;
    uint32_t k = 0, total = 0;
    unsigned long long slot = 0, x = 0, sum = 0, mism = 0;
    bool fresh = false, grown = false;
    unsigned at = 0;
    if (warp == 0) {
      slot = first + (unsigned long long)lane * gridDim.x;
      if (keep && keep[lane].sess >= 0) {
        const serve_lane l = keep[lane];
        sess = l.sess;
        k = l.k;
        total = l.total;
        x = l.x;
        sum = l.sum;
        mism = l.mism;
      } else if (slot < A.n_slots) {
        sess = __ldcg(&A.slot_session[slot]);
        fresh = sess < -1;
        if (fresh) sess = -2 - sess;
        if (sess >= 0) total = A.blocks[sess];
      }
      if (!keep && sess >= 0) {
        if (!fresh) {
          k = A.slot_k[slot];
          x = A.slot_acc[3 * slot];
          sum = A.slot_acc[3 * slot + 1];
          mism = A.slot_acc[3 * slot + 2];
        }
      }
      __syncwarp();
      const bool want = sess >= 0 && k < total;
      unsigned char *bp = serve_malloc<V>(h, A.block_bytes, want);
      __syncwarp();
      grown = want && bp;
      const unsigned gm = __ballot_sync(0xffffffffu, grown), wm = __ballot_sync(0xffffffffu, want);
      at = __popc(gm & lanemask_lt());
      if (grown) {
        A.tables[slot * A.max_blocks + k] = reinterpret_cast<unsigned long long>(bp);
        s_bp[at] = bp;
        s_key[at] = fmix32((A.seed + (uint32_t)sess) ^ (k * OURO_GOLD));
        s_sum[at] = 0;
        s_xor[at] = s_mism[at] = 0;
      }
      if (lane == 0) {
        s_n = __popc(gm);
        if (gm) atomicAdd(&A.ctl[5], (unsigned long long)__popc(gm));
        if (wm != gm) atomicAdd(&A.ctl[7], (unsigned long long)__popc(wm & ~gm));
      }
    }
    __syncthreads();
    const unsigned pieces = s_n * per;
    const unsigned long long pol = stream_policy();
    for (unsigned t = warp; t < pieces; t += nwarps) {
      const unsigned b = t / per, u0 = (t - b * per) * SERVE_PIECE;
      uint4 *u4 = reinterpret_cast<uint4 *>(s_bp[b]);
      const uint32_t key = s_key[b], end = min(units, u0 + SERVE_PIECE);
#pragma unroll 8
      for (uint32_t u = u0 + lane; u < end; u += 32) st_stream(u4 + u, pat4(key, 4 * u), pol);
    }
    __syncthreads();
    for (unsigned t = (warp + 1) % nwarps; t < pieces; t += nwarps) {
      const unsigned b = t / per, u0 = (t - b * per) * SERVE_PIECE;
      const uint4 *u4 = reinterpret_cast<const uint4 *>(s_bp[b]);
      const uint32_t key = s_key[b], end = min(units, u0 + SERVE_PIECE);
      payload_acc a;
      uint4 g[SERVE_PIECE / 32];
#pragma unroll
      for (unsigned r = 0; r < SERVE_PIECE / 32; ++r)
        if (u0 + 32 * r + lane < end) g[r] = ld_stream(u4 + u0 + 32 * r + lane, pol);
#pragma unroll
      for (unsigned r = 0; r < SERVE_PIECE / 32; ++r)
        if (u0 + 32 * r + lane < end) check4(g[r], pat4(key, 4 * (u0 + 32 * r + lane)), a);
      const unsigned ax = __reduce_xor_sync(0xffffffffu, a.x), am = __reduce_add_sync(0xffffffffu, a.mism);
      for (int o = 16; o; o >>= 1) a.s += __shfl_xor_sync(0xffffffffu, a.s, o);
      if (lane == 0) {
        atomicXor(&s_xor[b], ax);
        atomicAdd(&s_sum[b], a.s);
        if (am) atomicAdd(&s_mism[b], am);
      }
    }
    __syncthreads();
    if (warp == 0 && sess >= 0) {
      if (grown) {
        ++k;
        x ^= s_xor[at];
        sum += s_sum[at];
        mism += s_mism[at];
      }
      if (!keep || k >= total) A.slot_k[slot] = k;
      if (keep) {
        keep[lane].sess = k < total ? sess : -1;
        keep[lane].k = k;
        keep[lane].total = total;
        keep[lane].x = x;
        keep[lane].sum = sum;
        keep[lane].mism = mism;
      }
      if (k < total && !keep) {
        if (fresh) A.slot_session[slot] = sess;
        A.slot_acc[3 * slot] = x;
        A.slot_acc[3 * slot + 1] = sum;
        A.slot_acc[3 * slot + 2] = mism;
      } else if (k >= total) {   /* complete: report, release the slot (reused from the next step on), list it for freeing */
        A.sess_out[5ull * sess + 0] = x;
        A.sess_out[5ull * sess + 1] = sum;
        A.sess_out[5ull * sess + 2] = mism;
        A.sess_out[5ull * sess + 4] = step;
        atomicAdd(&A.ctl[6], (unsigned long long)k);
        atomicAdd(&A.ctl[3], 0ull - (unsigned long long)total);
        A.slot_session[slot] = -1;
        A.free_stack[atomicAdd(&A.ctl[8], 1ull)] = (uint32_t)slot;
        A.done_list[atomicAdd(&A.ctl[9 + (step & 1)], 1ull)] = (uint32_t)slot;
      }
    }
    __syncthreads();
  }
}

/* blocks of a finished session freed per task: one warp round, so that the
 * step's frees spread over as many warps as there are rounds of work */
constexpr uint32_t SERVE_FREE_TASK = 32;

/* Freeing: the listed sessions' blocks, in tasks of SERVE_FREE_TASK blocks; warp
 *     w takes tasks w, w + nwarps, ... (tasks are of equal size, so a static
 *     share balances without a shared counter): task c is piece
 *     c - (pieces of the earlier list entries) of the first entry whose
 *     running piece count passes c */
template <int V>
__device__ void serve_free(const serve_args &A, uint32_t step) {
  const unsigned lane = laneid();
  const unsigned long long nwarps = (gridDim.x * blockDim.x) >> 5;
  const ouro_heap_dev &h = A.h;
  const int cls = size_class(h, A.block_bytes);   /* of every block in the tables */
  const unsigned long long nl = *(volatile unsigned long long *)&A.ctl[9 + (step & 1)];
  for (unsigned long long c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;; c += nwarps) {
    unsigned long long before = 0;
    uint32_t slot = 0, nb = 0;
    bool found = false;
    for (unsigned long long i0 = 0; i0 < nl && !found; i0 += 32) {
      const unsigned long long i = i0 + lane;
      const uint32_t s_i = i < nl ? __ldcg(&A.done_list[i]) : 0;
      const uint32_t nb_i = i < nl ? __ldcg(&A.slot_k[s_i]) : 0;
      unsigned long long pc = (nb_i + SERVE_FREE_TASK - 1) / SERVE_FREE_TASK, incl = pc;
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, i < nl && before + incl > c);
      if (hit) {
        const int l = __ffs(hit) - 1;
        slot = __shfl_sync(0xffffffffu, s_i, l);
        nb = __shfl_sync(0xffffffffu, nb_i, l);
        before += __shfl_sync(0xffffffffu, incl - pc, l);
        found = true;
      } else {
        before += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    if (!found) break;
    const uint32_t b_lo = (uint32_t)(c - before) * SERVE_FREE_TASK, b_hi = min(nb, b_lo + SERVE_FREE_TASK);
    for (uint32_t b0 = b_lo; b0 < b_hi; b0 += 32) {
      const uint32_t b = b0 + lane;
      void *p = b < b_hi ? reinterpret_cast<void *>(__ldcg(&A.tables[(size_t)slot * A.max_blocks + b])) : nullptr;
      if (b < b_hi) free_v<V>(h, p, cls);
      __syncwarp();
    }
  }
}

/* The cooperative form: every step in one launch, phases separated by grid
 * barriers; block 0 stamps %globaltimer when a step begins to grow, when it
 * has grown and when its frees and the next admission are done. */
template <int V>
__global__ void __launch_bounds__(256, 2) k_serve(serve_args A) {
  unsigned epoch = 0;
  serve_init(A);
  if (!grid_barrier(A.ctl, gridDim.x, A.spin_limit, epoch)) return;
  if (A.steps) serve_admit(A, 0);
  if (!grid_barrier(A.ctl, gridDim.x, A.spin_limit, epoch)) return;
  const bool stamps = blockIdx.x == 0 && threadIdx.x == 0;
  __shared__ serve_lane lanes[32];
  serve_lane *keep = A.n_slots <= 32ull * gridDim.x ? lanes : nullptr;
  if (threadIdx.x < 32) lanes[threadIdx.x].sess = -1;
  for (uint32_t step = 0; step < A.steps; ++step) {
    if (stamps) A.step_ns[3 * step] = globaltimer();
    serve_grow<V>(A, step, keep);
    if (!grid_barrier(A.ctl, gridDim.x, A.spin_limit, epoch)) break;
    if (stamps) A.step_ns[3 * step + 1] = globaltimer();
    if (step + 1 < A.steps) serve_admit(A, step + 1);
    serve_free<V>(A, step);
    if (!grid_barrier(A.ctl, gridDim.x, A.spin_limit, epoch)) break;
    if (stamps) A.step_ns[3 * step + 2] = globaltimer();
  }
  if (keep && threadIdx.x < 32 && keep[threadIdx.x].sess >= 0) {   /* unfinished: the caller finds what still lives */
    const serve_lane &l = keep[threadIdx.x];
    const unsigned long long slot = blockIdx.x + (unsigned long long)threadIdx.x * gridDim.x;
    A.slot_session[slot] = l.sess;
    A.slot_k[slot] = l.k;
    A.slot_acc[3 * slot] = l.x;
    A.slot_acc[3 * slot + 1] = l.sum;
    A.slot_acc[3 * slot + 2] = l.mism;
  }
}

/* The per-launch form: one kernel per phase and step, in stream order.  A
 * phase kernel first stamps %globaltimer into step_ns[stamp] and, where
 * stamp2 >= 0, step_ns[stamp2]: the moment the previous phase had finished on
 * the whole grid. */
enum { PH_INIT, PH_ADMIT, PH_GROW, PH_FREE, PH_STAMP };

template <int V, int PH>
__global__ void __launch_bounds__(256, 2) k_serve_phase(serve_args A, uint32_t step, int stamp, int stamp2) {
  if (blockIdx.x == 0 && threadIdx.x == 0 && stamp >= 0) {
    const unsigned long long t = globaltimer();
    A.step_ns[stamp] = t;
    if (stamp2 >= 0) A.step_ns[stamp2] = t;
  }
  if (PH == PH_INIT) serve_init(A);
  if (PH == PH_ADMIT) serve_admit(A, step);
  if (PH == PH_GROW) serve_grow<V>(A, step, nullptr);
  if (PH == PH_FREE) {
    if (step + 1 < A.steps) serve_admit(A, step + 1);
    serve_free<V>(A, step);
  }
}

#if OURO_SHARD_ENTRIES
inline cudaStream_t S(void *s) { return reinterpret_cast<cudaStream_t>(s); }
#endif

}  // namespace

/* ------------------------------------------------------- per-form launcher */
namespace ouro {
namespace launch {

/* args: the kernel's serve_args, set up by ouro_serve */
template <int V>
ouro_status serve(const void *args, int blocks_per_sm, cudaStream_t s) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_serve<V>, 256, 0);
  if (blocks_per_sm > 0 && blocks_per_sm < per_sm) per_sm = blocks_per_sm;
  if (per_sm < 1) per_sm = 1;
  void *argv[] = {const_cast<void *>(args)};
  OURO_CUDA(cudaLaunchCooperativeKernel((const void *)k_serve<V>, dim3(per_sm * ouro::host::sm_count()), dim3(256),
                                        argv, 0, s));
  OURO_LAUNCHED();
  return OURO_OK;
}

/* the per-launch form: two launches per step (growth; freeing and the next
 * admission) plus the set-up, the first admission and a final stamp, in
 * stream order */
template <int V>
ouro_status serve_steps(const void *args, int blocks_per_sm, cudaStream_t s) {
  const serve_args &A = *static_cast<const serve_args *>(args);
  const int sms = ouro::host::sm_count();
  int grow_sm = 0, free_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&grow_sm, k_serve_phase<V, PH_GROW>, 256, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&free_sm, k_serve_phase<V, PH_FREE>, 256, 0);
  if (blocks_per_sm > 0) {
    grow_sm = std::min(grow_sm, blocks_per_sm);
    free_sm = std::min(free_sm, blocks_per_sm);
  }
  /* growth: a block per slot at most; slots: a thread per slot */
  const unsigned grow_g = (unsigned)std::max(1, (int)std::min<long long>((long long)grow_sm * sms, A.n_slots));
  const unsigned free_g = (unsigned)std::max(1, free_sm * sms);
  const unsigned slot_g = (unsigned)std::max(1u, std::min((A.n_slots + 255) / 256, 8u * sms));
  k_serve_phase<V, PH_INIT><<<slot_g, 256, 0, s>>>(A, 0, -1, -1);
  OURO_LAUNCHED();
  if (!A.steps) return OURO_OK;
  k_serve_phase<V, PH_ADMIT><<<1, 32, 0, s>>>(A, 0, -1, -1);
  OURO_LAUNCHED();
  for (uint32_t step = 0; step < A.steps; ++step) {
    k_serve_phase<V, PH_GROW><<<grow_g, 256, 0, s>>>(A, step, (int)(3 * step), step ? (int)(3 * step - 1) : -1);
    OURO_LAUNCHED();
    k_serve_phase<V, PH_FREE><<<free_g, 256, 0, s>>>(A, step, (int)(3 * step + 1), -1);
    OURO_LAUNCHED();
  }
  k_serve_phase<V, PH_STAMP><<<1, 32, 0, s>>>(A, 0, (int)(3 * A.steps - 1), -1);
  OURO_LAUNCHED();
  return OURO_OK;
}

#define INST_SERVE(PRE, V) PRE template ouro_status serve<V>(const void *, int, cudaStream_t);
#define INST_SERVE_STEPS(PRE, V) PRE template ouro_status serve_steps<V>(const void *, int, cudaStream_t);
OURO_SHARD_INSTANTIATE(INST_SERVE)
OURO_SHARD_INSTANTIATE(INST_SERVE_STEPS)

}  // namespace launch
}  // namespace ouro

#if OURO_SHARD_ENTRIES
namespace {
/* checks the arguments, resets the loop's state on the stream and fills A */
ouro_status serve_prepare(ouro_heap *H, const uint32_t *d_arrive_step, const uint32_t *d_blocks, uint32_t n_sessions,
                          uint32_t n_slots, uint32_t max_blocks, int *d_slot_session, uint32_t *d_slot_k,
                          unsigned long long *d_slot_acc, unsigned long long *d_tables,
                          unsigned long long *d_sess_out, unsigned long long *d_step_ns, unsigned long long *d_ctl,
                          uint32_t *d_free_stack, uint32_t steps, uint32_t seed, uint64_t cap_blocks,
                          uint32_t block_bytes, cudaStream_t s, serve_args &A) {
  if (!H || !d_arrive_step || !d_blocks || !d_slot_session || !d_slot_k || !d_slot_acc || !d_tables ||
      !d_sess_out || !d_step_ns || !d_ctl || !d_free_stack || n_slots == 0 || max_blocks == 0 || (block_bytes & 15) ||
      block_bytes == 0 || block_bytes > H->d.chunk_bytes)
    return OURO_EINVAL;
  OURO_CUDA(cudaMemsetAsync(d_slot_session, 0xFF, n_slots * sizeof(int), s));
  OURO_CUDA(cudaMemsetAsync(d_ctl, 0, 11 * 8, s));
  OURO_CUDA(cudaMemsetAsync(d_sess_out, 0xFF, (size_t)n_sessions * 5 * 8, s));
  A.h = H->d;
  A.arrive_step = d_arrive_step;
  A.blocks = d_blocks;
  A.n_sessions = n_sessions;
  A.n_slots = n_slots;
  A.max_blocks = max_blocks;
  A.slot_session = d_slot_session;
  A.slot_k = d_slot_k;
  A.slot_acc = d_slot_acc;
  A.tables = d_tables;
  A.sess_out = d_sess_out;
  A.step_ns = d_step_ns;
  A.ctl = d_ctl;
  A.free_stack = d_free_stack;
  A.done_list = d_free_stack + n_slots;
  A.steps = steps;
  A.seed = seed;
  A.cap_blocks = cap_blocks;
  A.block_bytes = block_bytes;
  A.spin_limit = 1u << 24;   /* barrier wait: each poll is a 32 ns nap and an L2 round trip, seconds in all */
  return OURO_OK;
}
}  // namespace

extern "C" ouro_status ouro_serve(ouro_heap *H, const uint32_t *d_arrive_step, const uint32_t *d_blocks,
                                  uint32_t n_sessions, uint32_t n_slots, uint32_t max_blocks, int *d_slot_session,
                                  uint32_t *d_slot_k, unsigned long long *d_slot_acc, unsigned long long *d_tables,
                                  unsigned long long *d_sess_out, unsigned long long *d_step_ns,
                                  unsigned long long *d_ctl, uint32_t *d_free_stack, uint32_t steps, uint32_t seed,
                                  uint64_t cap_blocks, uint32_t block_bytes, int blocks_per_sm, void *stream) {
  cudaStream_t s = S(stream);
  serve_args A;
  const ouro_status st = serve_prepare(H, d_arrive_step, d_blocks, n_sessions, n_slots, max_blocks, d_slot_session,
                                       d_slot_k, d_slot_acc, d_tables, d_sess_out, d_step_ns, d_ctl, d_free_stack,
                                       steps, seed, cap_blocks, block_bytes, s, A);
  if (st != OURO_OK) return st;
  int dev = 0, coop = 0;
  OURO_CUDA(cudaGetDevice(&dev));
  OURO_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return OURO_ENOTSUP;
  OURO_DISPATCH(H->d.variant, return ouro::launch::serve<V>(&A, blocks_per_sm, s));
}

extern "C" ouro_status ouro_serve_per_launch(ouro_heap *H, const uint32_t *d_arrive_step, const uint32_t *d_blocks,
                                             uint32_t n_sessions, uint32_t n_slots, uint32_t max_blocks,
                                             int *d_slot_session, uint32_t *d_slot_k, unsigned long long *d_slot_acc,
                                             unsigned long long *d_tables, unsigned long long *d_sess_out,
                                             unsigned long long *d_step_ns, unsigned long long *d_ctl,
                                             uint32_t *d_free_stack, uint32_t steps, uint32_t seed,
                                             uint64_t cap_blocks, uint32_t block_bytes, int blocks_per_sm,
                                             void *stream) {
  cudaStream_t s = S(stream);
  serve_args A;
  const ouro_status st = serve_prepare(H, d_arrive_step, d_blocks, n_sessions, n_slots, max_blocks, d_slot_session,
                                       d_slot_k, d_slot_acc, d_tables, d_sess_out, d_step_ns, d_ctl, d_free_stack,
                                       steps, seed, cap_blocks, block_bytes, s, A);
  if (st != OURO_OK) return st;
  OURO_DISPATCH(H->d.variant, return ouro::launch::serve_steps<V>(&A, blocks_per_sm, s));
}
#endif
