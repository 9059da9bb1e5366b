/*
 * Batch API and driver-round kernels.
 *
 * The paper's driver (Sec. 3 of arXiv 2504.18211) allocates, writes some
 * data, reads it back to check it, and frees, ten times over.  Two forms:
 *   - per launch: ouro_batch_malloc, ouro_pattern_write, ouro_pattern_check,
 *     ouro_batch_free (four kernels per round);
 *   - fused: ouro_round_fused, one kernel per round; the allocator state
 *     stays in L2 while every warp streams its own blocks.
 * Payload traffic is warp-cooperative: the 32 blocks of a warp are cut into
 * 16-byte units that the 32 lanes write and read in turn, so stores and
 * loads are 16-byte vectors that coalesce within each block.
 */
#include <type_traits>

#include "ouro_internal.cuh"
#include "ouro_payload.cuh"
#include "ouro_shard.cuh"

using namespace ouro::detail;

namespace {
/* ------------------------------------------------------------ batch API */
template <int V>
__global__ void k_batch_malloc(ouro_heap_dev h, const uint32_t *sizes, void **ptrs, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    ptrs[i] = malloc_v<V>(h, sizes[i]);
}

template <int V>
__global__ void k_batch_free(ouro_heap_dev h, void *const *ptrs, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    free_v<V, false>(h, ptrs[i]);   /* the blocks were written by earlier kernels */
}

/* Block-aggregated forms (page queues, not the deoptimised form): every
 * request of a block takes its offset in its class's share with one
 * shared-memory atomic, and one thread per class takes the whole block's
 * head (malloc) or tail (free) positions with a single global atomic, so
 * the hot queue counters see one atomic per class per block instead of one
 * per class per warp.  Statistics are counted once per class per block,
 * requests without a class among them: as one global reduction each they held
 * up the fence behind the slot loads (2^20 requests with 4 % of them: malloc
 * 24 us; the pass of malloc, id write, id check and free 117 us, 109 so).
 *
 * Each thread carries R requests (r * 256 + thread of the block's span, so
 * loads coalesce).  On plain-array queues a thread first tries all R of its
 * positions at once, pages and runs: R relaxed slot loads (malloc) or R
 * relaxed slot CASes (free) in flight together, behind one acquire / release
 * fence, instead of R chains of dependent round trips.  (With 2 % runs among
 * 2^20 requests every other warp went through the warp path for them: malloc
 * 28.6 us, 24 so.)  A position whose slot is not ready
 * (not produced yet, or its previous lap not consumed yet) goes through the
 * warp path with the position already taken, which waits, carves and
 * answers as ouro_malloc / ouro_free do. */
template <int R>
__device__ __forceinline__ void blk_reserve(const int (&cls)[R], unsigned long long (&pos)[R], unsigned *s_cnt) {
#pragma unroll
  for (int r = 0; r < R; ++r)   /* this request's offset in the block's share of its class */
    pos[r] = cls[r] >= 0 ? atomicAdd(&s_cnt[cls[r]], 1u) : 0u;
}

/* block of a taken item: a page id, or a run's first chunk, which is live again */
__device__ __forceinline__ void *blk_block(const ouro_heap_dev &h, int cls, unsigned item) {
  unsigned sh = 4u + cls;
  if (cls >= (int)h.n_classes) {
    h.chunk_cls[item] = (unsigned char)cls;
    sh = h.log2_chunk;
  }
  return h.base + ((size_t)item << sh);
}

/* Segments under a block's share of each class (virtualized queues, several
 * requests per thread): the share's positions are consecutive, so they lie in
 * at most BLK_SEGS segments unless the chunks are small.  One thread per class
 * and segment looks its segment up, all at once; every request then finds its
 * slot by offset, and the block counts its position events on a segment with
 * one atomic.  A share's further segments, and a segment that is not there
 * yet, are left to the warp path.  (3 * 2^18 requests of 64 B on a list,
 * malloc, write, check and free: 127 us with one request per thread and a
 * lookup per warp, 118 so.) */
constexpr unsigned BLK_SEGS = 4;
struct blk_segs {
  unsigned long long *cells[OURO_MAX_CLASSES][BLK_SEGS];   /* slot 0 of the segment; null: not known */
  unsigned events[OURO_MAX_CLASSES][BLK_SEGS];
  unsigned off0[OURO_MAX_CLASSES];                         /* offset of the share's first position */
  unsigned long long end[OURO_MAX_CLASSES];                /* consumers: the class's tail; further segments may not exist */
  unsigned retire;                                         /* classes with a segment to retire (lists) */
};

/* After the block's positions are taken; ends with a block barrier.  CREATE:
 * producers, who make missing segments and look ahead as va_slot / vl_slot do. */
template <int QF, bool CREATE>
__device__ void blk_segs_find(const ouro_heap_dev &h, blk_segs &sg, const unsigned *cnt, const unsigned long long *pos) {
  static_assert(OURO_MAX_CLASSES * BLK_SEGS <= 128, "a thread per class and segment of the smallest block");
  if (threadIdx.x < OURO_MAX_CLASSES * BLK_SEGS) {
    const unsigned c = threadIdx.x / BLK_SEGS, j = threadIdx.x % BLK_SEGS;
    unsigned long long *cells = nullptr;
    if (cnt[c]) {
      const unsigned long long s0 = pos[c] / h.seg_cap, s = s0 + j;
      const unsigned off0 = (unsigned)(pos[c] - s0 * h.seg_cap), end = off0 + cnt[c];   /* offsets from s0's slot 0 */
      if (j == 0) sg.off0[c] = off0;
      if (j * h.seg_cap < end && (CREATE || s * h.seg_cap < sg.end[c])) {
        const unsigned lo = j ? 0 : off0, hi = min(end - j * h.seg_cap, h.seg_cap);   /* the share in segment s: [lo, hi) */
        unsigned long long *cell = slot_at<QF>(h, (int)c, s * h.seg_cap + lo, CREATE);
        if (cell) {
          cells = cell - lo;
          const unsigned w = h.seg_cap >> 3;
          if (CREATE && lo < w && hi > w) {   /* the look-ahead of the positions just past 1/8 of the segment */
            if (QF == OURO_QF_VARRAY) va_prefetch(h, (int)c, (unsigned)s + 1);
            else vl_prefetch(h, (int)c, pack((unsigned)s, (unsigned)(((const unsigned char *)cell - h.base) >> h.log2_chunk)));
          }
        }
      }
    }
    sg.cells[c][j] = cells;
    sg.events[c][j] = 0;
    if (threadIdx.x == 0) sg.retire = 0;
  }
  __syncthreads();
}

/* slot of the request of rank `rank` in the block's share of class c, and its
 * segment j; null: not known */
__device__ __forceinline__ unsigned long long *blk_segs_slot(const ouro_heap_dev &h, const blk_segs &sg, int c,
                                                             unsigned rank, unsigned &j) {
  const unsigned off = sg.off0[c] + rank;
  j = off / h.seg_cap;
  return j < BLK_SEGS && sg.cells[c][j] ? sg.cells[c][j] + (off - j * h.seg_cap) : nullptr;
}

/* Counts the block's events and retires the segments that saw their last one.
 * Called by every thread after a block barrier. */
template <int QF>
__device__ void blk_segs_events(const ouro_heap_dev &h, blk_segs &sg) {
  if (threadIdx.x < OURO_MAX_CLASSES * BLK_SEGS) {
    const unsigned c = threadIdx.x / BLK_SEGS, j = threadIdx.x % BLK_SEGS, n = sg.events[c][j];
    if (n) {
      const unsigned x = (unsigned)(((const unsigned char *)sg.cells[c][j] - h.base) >> h.log2_chunk);
      if (atomicAdd(&seg_of(h, x)->done, n) + n == 2u * h.seg_cap) {
        __threadfence();
        if (QF == OURO_QF_LIST) atomicOr(&sg.retire, 1u << c);
        else va_retire(h, (int)c, x);
      }
    }
  }
  if (QF != OURO_QF_LIST) return;
  __syncthreads();
  for (unsigned rm = sg.retire, k = 0; rm; rm &= rm - 1, ++k)   /* a warp for each such class */
    if (k % (blockDim.x >> 5) == threadIdx.x >> 5) vl_advance_warp<OURO_VL_WIDE_BATCH>(h, __ffs(rm) - 1);
}

/* out of line: R copies of the warp path inlined spilled 2 KB a thread */
template <int V>
__device__ __noinline__ void *blk_malloc_rest(const ouro_heap_dev &h, int cls, unsigned long long pos) {
  return page_malloc<V, 1, true>(h, cls, 0xffffffffu, pos);
}
template <int V>
__device__ __noinline__ void blk_free_rest(const ouro_heap_dev &h, int cls, unsigned item, unsigned vmask,
                                           unsigned long long pos) {
  page_free<V, true>(h, cls, item, vmask, pos);
}

template <int V, int R>
__global__ void __launch_bounds__(256, 4) k_batch_malloc_blk(ouro_heap_dev h, const uint32_t *sizes, void **ptrs,
                                                             size_t n) {
  ouro::chain_begin();
  constexpr int QF = ouro_qform(V);
  constexpr bool RING = QF == OURO_QF_RING, SEGS = !RING && R > 1;
  __shared__ typename std::conditional<SEGS, blk_segs, char>::type sg;
  __shared__ unsigned s_cnt[OURO_MAX_CLASSES], s_ok[OURO_MAX_CLASSES];
  __shared__ unsigned long long s_pos[OURO_MAX_CLASSES];
  __shared__ unsigned long long *s_ring[OURO_MAX_CLASSES];
  __shared__ unsigned long long s_rmask[OURO_MAX_CLASSES];
  if (threadIdx.x < OURO_MAX_CLASSES) {
    s_ring[threadIdx.x] = h.cells + h.ring_off[threadIdx.x];
    s_rmask[threadIdx.x] = h.ring_mask[threadIdx.x];
  }
  __shared__ unsigned s_none[2];   /* requests without a class: OURO_ST_ZERO, OURO_ST_TOO_LARGE */
  if (threadIdx.x < 2) s_none[threadIdx.x] = 0;
  __syncthreads();
  const size_t span = (size_t)blockDim.x * R;
  for (size_t base = (size_t)blockIdx.x * span; base < n; base += (size_t)gridDim.x * span) {
    uint32_t sz[R];
    int cls[R];
    unsigned long long pos[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const size_t i = base + (size_t)r * blockDim.x + threadIdx.x;
      sz[r] = i < n ? sizes[i] : 0;
    }
    if (threadIdx.x < OURO_MAX_CLASSES) s_cnt[threadIdx.x] = s_ok[threadIdx.x] = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool act = base + (size_t)r * blockDim.x + threadIdx.x < n;
      cls[r] = act ? size_class(h, sz[r]) : -1;
      if (act && cls[r] < 0) atomicAdd(&s_none[sz[r] == 0 ? OURO_ST_ZERO : OURO_ST_TOO_LARGE], 1u);
    }
    __syncthreads();
    blk_reserve<R>(cls, pos, s_cnt);
    __syncthreads();
    if (threadIdx.x < OURO_MAX_CLASSES && s_cnt[threadIdx.x]) {
      if constexpr (SEGS) sg.end[threadIdx.x] = ld_rlx(&qh(h, threadIdx.x)->tail.v);
      s_pos[threadIdx.x] = atomicAdd(&qh(h, threadIdx.x)->head.v, (unsigned long long)s_cnt[threadIdx.x]);
    }
    __syncthreads();
    void *res[R];
    bool pend[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      res[r] = nullptr;
      pend[r] = cls[r] >= 0;
    }
    if constexpr (SEGS) {   /* fast path of virtualized queues: every position's slot at once */
      blk_segs_find<QF, false>(h, sg, s_cnt, s_pos);
      if (!h.checked) {
        unsigned long long v[R];
        unsigned j[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          unsigned long long *cell = pend[r] ? blk_segs_slot(h, sg, cls[r], (unsigned)pos[r], j[r]) : nullptr;
          v[r] = cell ? ld_rlx(cell) : 0ull;
          if (!cell) j[r] = BLK_SEGS;
        }
        fence_acq_rel();
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (!pend[r] || j[r] == BLK_SEGS) continue;
          const int d = slot_d(v[r], pos[r] + s_pos[cls[r]]);
          if (d == 1 || d == 2) {
            if (d == 1) res[r] = blk_block(h, cls[r], lo32(v[r]));
            atomicAdd(&sg.events[cls[r]][j[r]], 1u);
            pend[r] = false;
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (cls[r] >= 0) pos[r] += s_pos[cls[r]];
    if (RING && !h.checked) {   /* fast path: every position's slot at once */
      unsigned long long v[R];
#pragma unroll
      for (int r = 0; r < R; ++r)
        v[r] = pend[r] ? ld_rlx(s_ring[cls[r]] + (pos[r] & s_rmask[cls[r]])) : 0ull;
      fence_acq_rel();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!pend[r]) continue;
        const int d = slot_d(v[r], pos[r]);
        if (d == 1 || d == 2) {   /* an item, or the heap's null answer: take it, retire the slot */
          st_rlx(s_ring[cls[r]] + (pos[r] & s_rmask[cls[r]]), slot(pos[r] + s_rmask[cls[r]] + 1, 0));
          if (d == 1) res[r] = blk_block(h, cls[r], lo32(v[r]));
          pend[r] = false;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {   /* the rest: the warp path from the taken positions */
      if (!__any_sync(0xffffffffu, pend[r])) continue;
      void *q;
      if constexpr (SEGS) q = blk_malloc_rest<V>(h, pend[r] ? cls[r] : -1, pos[r]);
      else q = page_malloc<V, 1, true>(h, pend[r] ? cls[r] : -1, 0xffffffffu, pos[r]);
      if (pend[r]) res[r] = q;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const size_t i = base + (size_t)r * blockDim.x + threadIdx.x;
      if (i < n) ptrs[i] = res[r];
      if (res[r]) atomicAdd(&s_ok[cls[r]], 1u);
    }
    __syncthreads();
    if constexpr (SEGS) blk_segs_events<QF>(h, sg);
    if (threadIdx.x < OURO_MAX_CLASSES && s_cnt[threadIdx.x]) {
      stat_add(h, threadIdx.x, OURO_ST_MALLOC, s_ok[threadIdx.x]);
      stat_add(h, threadIdx.x, OURO_ST_FAILED, s_cnt[threadIdx.x] - s_ok[threadIdx.x]);
    }
    __syncthreads();
  }
  if (threadIdx.x < 2) stat_add(h, OURO_ROW_NONE, threadIdx.x, s_none[threadIdx.x]);
}

template <int V, int R>
__global__ void __launch_bounds__(256) k_batch_free_blk(ouro_heap_dev h, void *const *ptrs, size_t n) {
  ouro::chain_begin();
  constexpr int QF = ouro_qform(V);
  constexpr bool RING = QF == OURO_QF_RING, SEGS = !RING && R > 1;
  __shared__ typename std::conditional<SEGS, blk_segs, char>::type sg;
  __shared__ unsigned s_cnt[OURO_MAX_CLASSES];
  __shared__ unsigned long long s_pos[OURO_MAX_CLASSES];
  __shared__ unsigned long long *s_ring[OURO_MAX_CLASSES];
  __shared__ unsigned long long s_rmask[OURO_MAX_CLASSES];
  if (threadIdx.x < OURO_MAX_CLASSES) {
    s_ring[threadIdx.x] = h.cells + h.ring_off[threadIdx.x];
    s_rmask[threadIdx.x] = h.ring_mask[threadIdx.x];
  }
  const size_t span = (size_t)blockDim.x * R;
  for (size_t base = (size_t)blockIdx.x * span; base < n; base += (size_t)gridDim.x * span) {
    void *p[R];
    unsigned item[R];
    int cls[R];
    unsigned long long pos[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const size_t i = base + (size_t)r * blockDim.x + threadIdx.x;
      p[r] = i < n ? ptrs[i] : nullptr;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      item[r] = 0;
      cls[r] = free_locate<V>(h, p[r], item[r]);
    }
    if (threadIdx.x < OURO_MAX_CLASSES) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    blk_reserve<R>(cls, pos, s_cnt);
    __syncthreads();
    if (threadIdx.x < OURO_MAX_CLASSES && s_cnt[threadIdx.x]) {
      s_pos[threadIdx.x] = atomicAdd(&qh(h, threadIdx.x)->tail.v, (unsigned long long)s_cnt[threadIdx.x]);
      stat_add(h, threadIdx.x, OURO_ST_FREE, s_cnt[threadIdx.x]);
    }
    __syncthreads();
    bool pend[R];
    if constexpr (SEGS) blk_segs_find<QF, true>(h, sg, s_cnt, s_pos);
#pragma unroll
    for (int r = 0; r < R; ++r) pend[r] = cls[r] >= 0;
    if constexpr (SEGS) {   /* fast path of virtualized queues: one release fence, then every slot's exchange at once */
      unsigned long long old[R];
      unsigned j[R];
      fence_acq_rel();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        unsigned long long *cell = pend[r] ? blk_segs_slot(h, sg, cls[r], (unsigned)pos[r], j[r]) : nullptr;
        if (cell) old[r] = exch_rlx(cell, slot(pos[r] + s_pos[cls[r]] + 1, item[r]));
        else j[r] = BLK_SEGS;
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!pend[r] || j[r] == BLK_SEGS) continue;
        if (slot_d(old[r], pos[r] + s_pos[cls[r]]) >= 3) {   /* its consumer gave the position up */
          stat_add(h, cls[r], OURO_ST_REPUSH, 1);
          push_one<QF>(h, cls[r], item[r]);
        }
        atomicAdd(&sg.events[cls[r]][j[r]], 1u);
        pend[r] = false;
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (cls[r] >= 0) pos[r] += s_pos[cls[r]];
    if (RING) {   /* fast path: one release fence, then every slot's CAS at once */
      unsigned long long old[R];
      fence_acq_rel();
#pragma unroll
      for (int r = 0; r < R; ++r)
        old[r] = pend[r] ? cas_rlx(s_ring[cls[r]] + (pos[r] & s_rmask[cls[r]]), slot(pos[r], 0), slot(pos[r] + 1, item[r]))
                         : 0ull;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (pend[r] && old[r] == slot(pos[r], 0)) pend[r] = false;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {   /* the rest: the warp path at the taken positions */
      const unsigned vmask = __ballot_sync(0xffffffffu, pend[r]);
      if (!pend[r]) continue;
      if constexpr (SEGS) blk_free_rest<V>(h, cls[r], item[r], vmask, pos[r]);
      else page_free<V, true>(h, cls[r], item[r], vmask, pos[r]);
    }
    __syncthreads();
    if constexpr (SEGS) {
      blk_segs_events<QF>(h, sg);
      __syncthreads();
    }
  }
}

/* Block-aggregated batch free for chunk queues (not the deoptimised form):
 * each request sets its page bit and counts it back on its chunk with its
 * warp, as a single free does (one atomicOr per (chunk, word) group, one
 * count atomic per chunk group), all R of a thread in flight together; the
 * chunks whose count that lifted, and the freed runs, take their rank in their
 * class's share of the block with one shared-memory atomic, and one thread per
 * class takes the block's tail positions with a single global atomic.  Per
 * warp, those tail atomics piled up on the class of one page per chunk, where
 * every free lifts a chunk.  On plain arrays all R slots of a thread are then
 * filled behind one fence; a slot that is not ready, and the slots of
 * virtualized queues, take the warp path at the position already taken.
 * Statistics once per class per block.  (300,007 mixed requests, 2 % of them
 * runs that each went through the warp path, malloc to free: 105 us, 98 with
 * this and the malloc below.) */
template <int V, int R>
__global__ void __launch_bounds__(256) k_batch_free_cblk(ouro_heap_dev h, void *const *ptrs, size_t n) {
  ouro::chain_begin();
  constexpr bool RING = ouro_qform(V) == OURO_QF_RING;
  __shared__ unsigned s_cnt[OURO_MAX_CLASSES], s_free[OURO_MAX_CLASSES];
  __shared__ unsigned long long s_pos[OURO_MAX_CLASSES];
  const size_t span = (size_t)blockDim.x * R;
  for (size_t base = (size_t)blockIdx.x * span; base < n; base += (size_t)gridDim.x * span) {
    void *p[R];
    unsigned item[R], x[R];
    int cls[R];
    bool put[R];
    unsigned long long pos[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const size_t i = base + (size_t)r * blockDim.x + threadIdx.x;
      p[r] = i < n ? ptrs[i] : nullptr;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      item[r] = 0;
      cls[r] = free_locate<V>(h, p[r], item[r]);   /* a run is marked free here */
    }
    if (threadIdx.x < OURO_MAX_CLASSES) s_cnt[threadIdx.x] = s_free[threadIdx.x] = 0;
    __syncthreads();
    int pc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) pc[r] = cls[r] < (int)h.n_classes ? cls[r] : -1;
    chunk_release_n<R, false>(h, pc, p, 0xffffffffu, x, put);   /* pc: -1 on a double free */
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (cls[r] >= (int)h.n_classes) {            /* a run: its first chunk goes to its class queue */
        put[r] = true;
        x[r] = item[r];
      } else {
        cls[r] = pc[r];
      }
      if (cls[r] >= 0) atomicAdd(&s_free[cls[r]], 1u);
      pos[r] = put[r] ? atomicAdd(&s_cnt[cls[r]], 1u) : 0u;
    }
    __syncthreads();
    if (threadIdx.x < OURO_MAX_CLASSES) {
      if (s_cnt[threadIdx.x])
        s_pos[threadIdx.x] = atomicAdd(&qh(h, threadIdx.x)->tail.v, (unsigned long long)s_cnt[threadIdx.x]);
      if (s_free[threadIdx.x]) stat_add(h, threadIdx.x, OURO_ST_FREE, s_free[threadIdx.x]);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (put[r]) pos[r] += s_pos[cls[r]];
    if (RING) {
      unsigned long long old[R];
      fence_acq_rel();
#pragma unroll
      for (int r = 0; r < R; ++r)
        old[r] = put[r] ? cas_rlx(ring_slot(h, cls[r], pos[r]), slot(pos[r], 0), slot(pos[r] + 1, x[r])) : 0ull;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (put[r] && old[r] == slot(pos[r], 0)) put[r] = false;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {   /* the rest: the warp path at the taken positions */
      const unsigned vmask = __ballot_sync(0xffffffffu, put[r]);
      if (put[r]) page_free<V, true>(h, cls[r], x[r], vmask, pos[r]);
    }
    __syncthreads();
  }
}

/* Block-aggregated batch malloc for chunk queues (not the deoptimised
 * form): every request takes its rank in its class's share of the block
 * with one shared-memory atomic; the shares are cut into tasks of at most
 * 32 whole chunks' pages (what one round of chunk_acquire serves from a
 * queue of whole chunks: 32 queue positions, each lane reserving and
 * claiming its chunk's part), and the block's warps take the tasks in turn,
 * classes with the fewest pages per chunk first, into a shared-memory page
 * list from which every request takes the page of its rank.  A class of
 * one page per chunk thus spreads over several warps instead of costing
 * one warp a round per 32 requests while the others wait at the barrier.
 * Requests above one chunk (runs) take their queue positions for the whole
 * block too; on plain arrays a thread tries all its runs' slots together, and
 * what is not ready takes the warp path of page_malloc at the position already
 * taken.  Statistics once per class per block.  (300,007 mixed requests, 2 %
 * of them runs that each went through the warp path, malloc to free: 105 us, 98
 * with this and the free above.) */
/* (registers: the compiler's choice, but for the list, where it may settle at 80
 * with 2 KB a thread spilled: 311,304 mixed requests 139 us, 134 at 128) */
template <int V, int R>
__global__ void __launch_bounds__(256, V == OURO_CHUNK_VLIST ? 2 : 0) k_batch_malloc_cblk(ouro_heap_dev h, const uint32_t *sizes, void **ptrs,
                                                           size_t n) {
  ouro::chain_begin();
  constexpr bool RING = ouro_qform(V) == OURO_QF_RING;
  static_assert(256 * R < 2048, "task offsets and counts are 11-bit fields");
  constexpr unsigned MAX_TASKS = (256 * R) / 32 + OURO_MAX_CLASSES;   /* sum over classes of ceil(share / part) */
  __shared__ unsigned s_cnt[OURO_MAX_CLASSES], s_base[OURO_MAX_CLASSES], s_ok[OURO_MAX_CLASSES];
  __shared__ unsigned s_items[256 * R];
  __shared__ unsigned s_task[MAX_TASKS];   /* class | offset << 5 | count << 16 */
  __shared__ unsigned s_ntask;
  __shared__ unsigned long long s_pos[OURO_MAX_CLASSES];   /* runs: head positions */
  __shared__ unsigned s_none[2];   /* requests without a class: OURO_ST_ZERO, OURO_ST_TOO_LARGE */
  if (threadIdx.x < 2) s_none[threadIdx.x] = 0;
  __syncthreads();
  const size_t span = (size_t)blockDim.x * R;
  const unsigned warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  for (size_t base = (size_t)blockIdx.x * span; base < n; base += (size_t)gridDim.x * span) {
    uint32_t sz[R];
    int cls[R];
    unsigned long long pos[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const size_t i = base + (size_t)r * blockDim.x + threadIdx.x;
      sz[r] = i < n ? sizes[i] : 0;
      cls[r] = i < n ? size_class(h, sz[r]) : -1;
      if (i < n && cls[r] < 0) atomicAdd(&s_none[sz[r] == 0 ? OURO_ST_ZERO : OURO_ST_TOO_LARGE], 1u);
    }
    if (threadIdx.x < OURO_MAX_CLASSES) s_cnt[threadIdx.x] = s_ok[threadIdx.x] = 0;
    __syncthreads();
    int pc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) pc[r] = cls[r] < (int)h.n_classes ? cls[r] : -1;
    blk_reserve<R>(cls, pos, s_cnt);
    __syncthreads();
    if (threadIdx.x >= h.n_classes && threadIdx.x < OURO_MAX_CLASSES && s_cnt[threadIdx.x])
      s_pos[threadIdx.x] = atomicAdd(&qh(h, threadIdx.x)->head.v, (unsigned long long)s_cnt[threadIdx.x]);
    if (threadIdx.x == 0) {
      unsigned acc = 0, nt = 0;
      for (unsigned c = 0; c < h.n_classes; ++c) {
        s_base[c] = acc;
        acc += s_cnt[c];
      }
      for (int c = (int)h.n_classes - 1; c >= 0; --c) {
        const unsigned part = 32u << (h.log2_chunk - 4 - c);
        for (unsigned o = 0; o < s_cnt[c]; o += part)
          s_task[nt++] = (unsigned)c | (o << 5) | (min(part, s_cnt[c] - o) << 16);
      }
      s_ntask = nt;
    }
    __syncthreads();
    for (unsigned t = warp; t < s_ntask; t += nwarps) {
      const unsigned tk = s_task[t], c = tk & 31u, cnt = tk >> 16;
      unsigned *out = s_items + s_base[c] + ((tk >> 5) & 2047u);
      const unsigned got = chunk_acquire<V>(h, (int)c, cnt, out);
      for (unsigned i = got + lane; i < cnt; i += 32) out[i] = OURO_NIL;   /* the heap ran out: null answers */
    }
    __syncthreads();
    void *res[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      res[r] = nullptr;
      if (pc[r] >= 0) {
        const unsigned item = s_items[s_base[pc[r]] + pos[r]];
        if (item != OURO_NIL) {
          res[r] = h.base + ((size_t)item << (4 + pc[r]));
          atomicAdd(&s_ok[pc[r]], 1u);
        }
      }
    }
    bool run[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      run[r] = cls[r] >= (int)h.n_classes;
      if (run[r]) pos[r] += s_pos[cls[r]];
    }
    if (RING) {   /* runs above one chunk: every position's slot at once */
      unsigned long long v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = run[r] ? ld_rlx(ring_slot(h, cls[r], pos[r])) : 0ull;
      fence_acq_rel();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!run[r]) continue;
        const int d = slot_d(v[r], pos[r]);
        if (d == 1 || d == 2) {
          st_rlx(ring_slot(h, cls[r], pos[r]), slot(pos[r] + h.ring_mask[cls[r]] + 1, 0));
          if (d == 1) {
            h.chunk_cls[lo32(v[r])] = (unsigned char)cls[r];
            res[r] = h.base + ((size_t)lo32(v[r]) << h.log2_chunk);
            atomicAdd(&s_ok[cls[r]], 1u);
          }
          run[r] = false;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {   /* the rest: the warp path from the taken positions */
      if (!__any_sync(0xffffffffu, run[r])) continue;
      void *q = page_malloc<V, 1, true>(h, run[r] ? cls[r] : -1, 0xffffffffu, pos[r]);
      if (run[r]) {
        res[r] = q;
        if (q) atomicAdd(&s_ok[cls[r]], 1u);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const size_t i = base + (size_t)r * blockDim.x + threadIdx.x;
      if (i < n) ptrs[i] = res[r];
    }
    __syncthreads();
    if (threadIdx.x < OURO_MAX_CLASSES && s_cnt[threadIdx.x]) {
      stat_add(h, threadIdx.x, OURO_ST_MALLOC, s_ok[threadIdx.x]);
      stat_add(h, threadIdx.x, OURO_ST_FAILED, s_cnt[threadIdx.x] - s_ok[threadIdx.x]);
    }
    __syncthreads();
  }
  if (threadIdx.x < 2) stat_add(h, OURO_ROW_NONE, threadIdx.x, s_none[threadIdx.x]);
}

/* mode 0 of k_pattern: one word per block, a lane each; a thread's four
 * pointers, then its four words, in flight together.  Every word is a sector
 * of its own, so what bounds it is scattered sectors, not bytes. */
template <int OP>
__device__ __forceinline__ void pattern_ids(void *const *ptrs, size_t n, payload_acc &a, unsigned long long &nulls) {
  const size_t threads = (size_t)gridDim.x * blockDim.x;
  for (size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += 4 * threads) {
    uint32_t *p[4];
    uint32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) p[k] = i0 + k * threads < n ? static_cast<uint32_t *>(ptrs[i0 + k * threads]) : nullptr;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (OP & PAY_WRITE) {
        if (p[k]) *p[k] = (uint32_t)(i0 + k * threads);
      } else {
        v[k] = p[k] ? __ldcg(p[k]) : 0u;
      }
    }
    if (OP & PAY_CHECK) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (p[k]) {
          a.mism += v[k] != (uint32_t)(i0 + k * threads);
          a.fold(v[k]);
          a.words++;
        } else if (i0 + k * threads < n) {
          nulls++;
        }
      }
    }
  }
}

/* The requests are cut into tasks: the first `heads` of them of 32 requests,
 * the rest of `task` requests (a power of two of at most 32).  The tasks are
 * dealt to the blocks in turn, and a block's warps pull the block's tasks from
 * a shared-memory counter: long tasks first, which share a row of small blocks
 * among 32 requests, short ones last, so that the warps end together.  With
 * fixed 32-request strides a warp had 3 or 4 of them at 2^20 requests and the
 * kernel waited for the fours. */
template <int OP>
__global__ void __launch_bounds__(256) k_pattern(void *const *ptrs, const uint32_t *sizes, size_t n, uint32_t seed,
                                                 int mode, size_t heads, unsigned task, ouro_check *out) {
  ouro::chain_begin();
  __shared__ unsigned s_next;
  if (threadIdx.x == 0) s_next = 0;
  __syncthreads();
  payload_acc a;
  unsigned long long nulls = 0;
  if (mode == 0) {
    pattern_ids<OP>(ptrs, n, a, nulls);
  } else {
    const unsigned lane = threadIdx.x & 31;
    const size_t tasks = heads + (n - 32 * heads + task - 1) / task;
    for (;;) {
      unsigned t = 0;
      if (lane == 0) t = atomicAdd(&s_next, 1u);
      t = __shfl_sync(0xffffffffu, t, 0);
      const size_t k = (size_t)t * gridDim.x + blockIdx.x;
      if (k >= tasks) break;
      const size_t i = (k < heads ? 32 * k : 32 * heads + (k - heads) * task) + lane;
      const bool mine = lane < (k < heads ? 32u : task) && i < n;
      unsigned char *p = mine ? static_cast<unsigned char *>(ptrs[i]) : nullptr;
      const uint32_t sz = mine ? sizes[i] : 0;
      if (mine && !p) nulls++;
      warp_payload<OP>(p, sz, (uint32_t)i, seed, 1, a);
    }
  }
  if (OP & PAY_CHECK) flush_acc(a, nulls, out);
}

/* A fused round's tasks past the warps' first ones: drawn from a counter in the
 * launch's slot, or without one in the half of *out's xor64 that stays zero. */
struct round_draws {
  unsigned long long first = 0;   /* the first request that is drawn for */
  unsigned *next;
  unsigned count = 0;             /* draws in all; 0: none */
  round_draws(size_t n, unsigned task, unsigned warps, work_slot *work, ouro_check *out) {
    first = (unsigned long long)warps * task;
    if (first < n) count = (unsigned)((n - first + task - 1) / task) + warps;
    next = work ? &work->next : reinterpret_cast<unsigned *>(&out->xor64) + 1;
  }
};

/* one whole round per thread: malloc, write, read back, free.  Warps take
 * `task` requests (a power of two of at most 32) at a time: warp w of the
 * grid the w-th task, then tasks from the launch's counter, so blocks of
 * uneven sizes balance across warps and the round ends within one task of
 * the last byte.  Where tasks are drawn at all, every warp draws until there
 * is none left, so the number of draws is known and the last one leaves the
 * counter zero.  The lanes past `task` ask for nothing but help their
 * warp's carves and payload.  STAGE: the warp's freed pages serve its next
 * mallocs of the same class from shared memory (heap option `staging`). */
#ifndef OURO_FUSED_MIN_BLOCKS
#define OURO_FUSED_MIN_BLOCKS 4   /* resident blocks of 256 per SM the fused round is compiled for */
#endif
/* chunk queues: their larger malloc path gets 2 blocks of 256 per SM
 * (128 registers a thread) instead of spilling at 64 */
template <int V, bool STAGE>
__global__ void __launch_bounds__(256, ouro_page_queues(V) ? OURO_FUSED_MIN_BLOCKS : 2) k_round_fused(ouro_heap_dev h, const uint32_t *sizes, size_t n,
                                                     uint32_t seed, int mode, unsigned task, ouro_check *out,
                                                     void **ptrs, work_slot *work, round_draws draw) {
  ouro::chain_begin();
  __shared__ ouro_block_ctx<8> ctx;
  if (STAGE) ouro_block_begin(ctx);
  payload_acc a;
  unsigned long long nulls = 0;
  const unsigned lane = threadIdx.x & 31;
  unsigned long long base = (unsigned long long)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * task;
  while (base < n) {
    const size_t i = base + lane;
    const bool mine = lane < task && i < n;
    const uint32_t sz = mine ? sizes[i] : 0;
    unsigned char *p;
    if (STAGE) p = static_cast<unsigned char *>(stage_malloc_v<V>(ctx, h, sz, mine));
    else p = static_cast<unsigned char *>(malloc_v<V>(h, sz, mine));
    if (mine) {
      if (!p) nulls++;
      if (ptrs) ptrs[i] = p;
    }
    __syncwarp();
    warp_payload<PAY_FUSED, plain_payload(V, STAGE), pace_payload(V, STAGE)>(p, sz, (uint32_t)i, seed, mode, a,
                                                                             task >= 16);
    __syncwarp();
    /* staged: the class of each block is known here, so the free skips the
     * chunk-table lookup (one L2 round trip per task off the warp's chain) */
    if (STAGE) ouro::detail::stage_free<V, 8>(ctx, h, p, __activemask(), p ? size_class(h, sz) : -1);
    else free_v<V>(h, p);
    __syncwarp();
    if (!draw.count) break;
    if (lane == 0) {
      const unsigned d = atomicAdd(draw.next, 1u);
      base = draw.first + (unsigned long long)d * task;
      if (d == draw.count - 1) *draw.next = 0;
    }
    base = __shfl_sync(0xffffffffu, base, 0);
  }
  if (STAGE) ouro_block_end_v<V>(ctx, h);
  finish_acc(a, nulls, work, out);
}

#if OURO_SHARD_ENTRIES
inline cudaStream_t S(void *s) { return reinterpret_cast<cudaStream_t>(s); }
#endif

template <typename K>
int occupancy_grid(K kernel, int block) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0);
  if (per_sm < 1) per_sm = 1;
  return per_sm * ouro::host::sm_count();
}

/* the largest power of two up to 32 that leaves every one of `warps` warps
 * `per` tasks of n requests (1 at least) */
inline unsigned task_size(size_t n, size_t warps, int per) {
  unsigned t = 1;
  while (t < 32 && 2 * t * warps * per <= n) t *= 2;
  return t;
}

inline int grid_for(size_t n, int block, int cap) {
  size_t g = (n + block - 1) / block;
  if (g < 1) g = 1;
  return (int)(g < (size_t)cap ? g : (size_t)cap);
}

#if OURO_SHARD_ENTRIES
/* How k_pattern cuts n requests: whole rounds of 32-request tasks for all
 * resident warps while they cover at most 7/8 of the requests, then tasks
 * that give every warp about four; a batch with less than a round, tasks of
 * an eighth of a warp's share (1024 blocks of 1000 B: one each).  Measured on
 * malloc + write + check + free of 2^20 size-sweep requests: fixed strides of
 * 32 697 us; all tasks of 32 / 16 / 8 / 4 requests 636 / 622 / 609 / 607; so
 * 607.  3 * 2^18 blocks of 64 B with all tasks of 8: 21 us each way, bound by
 * the instructions per task; so 17 and 20. */
struct pattern_shape {
  size_t heads = 0;
  unsigned task = 32;
  int grid;
  pattern_shape(size_t n, int mode, int block, int cap) {
    const size_t warps = (size_t)cap * (block / 32);
    size_t tasks = (n + 31) / 32;
    if (mode) {
      heads = n / 8 * 7 / (32 * warps) * warps;
      task = task_size(n - 32 * heads, warps, heads ? 4 : 8);
      tasks = heads + (n - 32 * heads + task - 1) / task;
    }
    grid = grid_for(tasks * 32, block, cap);
  }
};
#endif

}  // namespace

/* ------------------------------------------------------- per-form launchers */
namespace ouro {
namespace launch {

/* Requests per thread of the block-aggregated kernels: four (their slots are
 * tried together) once a batch fills every SM with four per thread; one
 * otherwise, so that a small batch still spreads over many blocks. */
constexpr int BLK_WIDE = 4;
static_assert(BLK_WIDE <= (int)OURO_BATCH_POS, "the queues' slack counts on it");
inline bool blk_wide(size_t n) { return n >= (size_t)BLK_WIDE * 256 * ouro::host::sm_count(); }
/* The plain-array batch free takes eight requests per thread in blocks of
 * 128 once a batch fills every SM with four such blocks: a 2^20 batch then
 * runs as one wave (1024 blocks, at most 56 registers a thread). */
constexpr int FREE_WIDE = 8, FREE_BLOCK = 128;
inline bool free_wide(size_t n) { return n >= (size_t)FREE_WIDE * FREE_BLOCK * 4 * ouro::host::sm_count(); }

template <int V>
ouro_status batch_malloc(ouro_heap *H, const uint32_t *d_sizes, void **d_ptrs, size_t n, cudaStream_t s) {
  const int block = 256;
  if constexpr (ouro_page_queues(V)) {
    if (!H->d.deopt) {
      if (blk_wide(n)) {
        ouro::host::launch_chained(k_batch_malloc_blk<V, BLK_WIDE>, grid_for((n + BLK_WIDE - 1) / BLK_WIDE, block, 1 << 20), block, s,
                                       H->d, d_sizes, d_ptrs, n);
        OURO_LAUNCHED();
        return OURO_OK;
      }
      ouro::host::launch_chained(k_batch_malloc_blk<V, 1>, grid_for(n, block, 1 << 20), block, s,
                                       H->d, d_sizes, d_ptrs, n);
      OURO_LAUNCHED();
      return OURO_OK;
    }
  }
  if constexpr (!ouro_page_queues(V)) {
    if (!H->d.deopt) {
      if (blk_wide(n))
        ouro::host::launch_chained(k_batch_malloc_cblk<V, BLK_WIDE>, grid_for((n + BLK_WIDE - 1) / BLK_WIDE, block, 1 << 20), block, s,
                                       H->d, d_sizes, d_ptrs, n);
      else
        ouro::host::launch_chained(k_batch_malloc_cblk<V, 1>, grid_for(n, block, 1 << 20), block, s,
                                       H->d, d_sizes, d_ptrs, n);
      OURO_LAUNCHED();
      return OURO_OK;
    }
  }
  k_batch_malloc<V><<<grid_for(n, block, 1 << 20), block, 0, s>>>(H->d, d_sizes, d_ptrs, n);
  OURO_LAUNCHED();
  return OURO_OK;
}

template <int V>
ouro_status batch_free(ouro_heap *H, void *const *d_ptrs, size_t n, cudaStream_t s) {
  const int block = 256;
  if constexpr (ouro_page_queues(V)) {
    if (!H->d.deopt) {
      if constexpr (ouro_qform(V) == OURO_QF_RING) {
        if (free_wide(n)) {
          ouro::host::launch_chained(k_batch_free_blk<V, FREE_WIDE>, grid_for((n + FREE_WIDE - 1) / FREE_WIDE, FREE_BLOCK, 1 << 20), FREE_BLOCK, s,
                                       H->d, d_ptrs, n);
          OURO_LAUNCHED();
          return OURO_OK;
        }
      }
      if (blk_wide(n)) {
        ouro::host::launch_chained(k_batch_free_blk<V, BLK_WIDE>, grid_for((n + BLK_WIDE - 1) / BLK_WIDE, block, 1 << 20), block, s,
                                       H->d, d_ptrs, n);
        OURO_LAUNCHED();
        return OURO_OK;
      }
      ouro::host::launch_chained(k_batch_free_blk<V, 1>, grid_for(n, block, 1 << 20), block, s,
                                       H->d, d_ptrs, n);
      OURO_LAUNCHED();
      return OURO_OK;
    }
  }
  if constexpr (!ouro_page_queues(V)) {
    if (!H->d.deopt) {
      if (blk_wide(n))
        ouro::host::launch_chained(k_batch_free_cblk<V, BLK_WIDE>, grid_for((n + BLK_WIDE - 1) / BLK_WIDE, block, 1 << 20), block, s,
                                       H->d, d_ptrs, n);
      else
        ouro::host::launch_chained(k_batch_free_cblk<V, 1>, grid_for(n, block, 1 << 20), block, s,
                                       H->d, d_ptrs, n);
      OURO_LAUNCHED();
      return OURO_OK;
    }
  }
  k_batch_free<V><<<grid_for(n, block, 1 << 20), block, 0, s>>>(H->d, d_ptrs, n);
  OURO_LAUNCHED();
  return OURO_OK;
}

template <int V, bool STAGE>
ouro_status round_fused_form(ouro_heap *H, const uint32_t *d_sizes, size_t n, uint32_t seed, int mode,
                             ouro_check *d_out, void **d_ptrs, void *work, cudaStream_t s) {
  const int block = 256, cap = occupancy_grid(k_round_fused<V, STAGE>, block);
  const unsigned task = ouro::host::round_task(n, (size_t)cap * (block / 32), ouro_page_queues(V), STAGE);
  const int grid = grid_for((n + task - 1) / task * 32, block, cap);
  work_slot *slot = static_cast<work_slot *>(work);
  ouro::host::launch_chained(k_round_fused<V, STAGE>, grid, block, s, H->d, d_sizes, n, seed, mode, task, d_out,
                             d_ptrs, slot, round_draws(n, task, grid * (block / 32), slot, d_out));
  OURO_LAUNCHED();
  return OURO_OK;
}

template <int V>
ouro_status round_fused(ouro_heap *H, const uint32_t *d_sizes, size_t n, uint32_t seed, int mode, ouro_check *d_out,
                        void **d_ptrs, void *work, cudaStream_t s) {
  return H->d.staging ? round_fused_form<V, true>(H, d_sizes, n, seed, mode, d_out, d_ptrs, work, s)
                      : round_fused_form<V, false>(H, d_sizes, n, seed, mode, d_out, d_ptrs, work, s);
}

#define INST_BATCH_MALLOC(PRE, V) \
  PRE template ouro_status batch_malloc<V>(ouro_heap *, const uint32_t *, void **, size_t, cudaStream_t);
#define INST_BATCH_FREE(PRE, V) \
  PRE template ouro_status batch_free<V>(ouro_heap *, void *const *, size_t, cudaStream_t);
#define INST_ROUND_FUSED(PRE, V)                                                                                 \
  PRE template ouro_status round_fused<V>(ouro_heap *, const uint32_t *, size_t, uint32_t, int, ouro_check *, \
                                          void **, void *, cudaStream_t);
OURO_SHARD_INSTANTIATE(INST_BATCH_MALLOC)
OURO_SHARD_INSTANTIATE(INST_BATCH_FREE)
OURO_SHARD_INSTANTIATE(INST_ROUND_FUSED)

}  // namespace launch
}  // namespace ouro

#if OURO_SHARD_ENTRIES
/* ------------------------------------------------------------- C entries */
extern "C" ouro_status ouro_batch_malloc(ouro_heap *H, const uint32_t *d_sizes, void **d_ptrs, size_t n,
                                         void *stream) {
  if (!H || (n && (!d_sizes || !d_ptrs))) return OURO_EINVAL;
  if (!n) return OURO_OK;
  OURO_DISPATCH(H->d.variant, return ouro::launch::batch_malloc<V>(H, d_sizes, d_ptrs, n, S(stream)));
}

extern "C" ouro_status ouro_batch_free(ouro_heap *H, void *const *d_ptrs, size_t n, void *stream) {
  if (!H || (n && !d_ptrs)) return OURO_EINVAL;
  if (!n) return OURO_OK;
  OURO_DISPATCH(H->d.variant, return ouro::launch::batch_free<V>(H, d_ptrs, n, S(stream)));
}

extern "C" ouro_status ouro_pattern_write(void *const *d_ptrs, const uint32_t *d_sizes, size_t n, uint32_t seed,
                                          int mode, void *stream) {
  if (n && (!d_ptrs || !d_sizes)) return OURO_EINVAL;
  if (mode != 0 && mode != 1) return OURO_EINVAL;
  if (!n) return OURO_OK;
  const int block = 256;
  const pattern_shape sh(n, mode, block, occupancy_grid(k_pattern<PAY_WRITE>, block));
  ouro::host::launch_chained(k_pattern<PAY_WRITE>, sh.grid, block, S(stream), d_ptrs, d_sizes, n, seed, mode, sh.heads, sh.task, nullptr);
  OURO_LAUNCHED();
  return OURO_OK;
}

extern "C" ouro_status ouro_pattern_check(void *const *d_ptrs, const uint32_t *d_sizes, size_t n, uint32_t seed,
                                          int mode, ouro_check *d_out, void *stream) {
  if (!d_out || (n && (!d_ptrs || !d_sizes))) return OURO_EINVAL;
  if (mode != 0 && mode != 1) return OURO_EINVAL;
  OURO_CUDA(cudaMemsetAsync(d_out, 0, sizeof(ouro_check), S(stream)));
  if (!n) return OURO_OK;
  const int block = 256;
  const pattern_shape sh(n, mode, block, occupancy_grid(k_pattern<PAY_CHECK>, block));
  ouro::host::launch_chained(k_pattern<PAY_CHECK>, sh.grid, block, S(stream), d_ptrs, d_sizes, n, seed, mode, sh.heads, sh.task, d_out);
  OURO_LAUNCHED();
  return OURO_OK;
}

namespace ouro {
namespace host {
ouro_status round_fused_on(ouro_heap *H, const uint32_t *d_sizes, size_t n, uint32_t seed, int mode, ouro_check *d_out,
                           void **d_ptrs, void *work, cudaStream_t s) {
  if (!n || !work) OURO_CUDA(cudaMemsetAsync(d_out, 0, sizeof(ouro_check), s));
  if (!n) return OURO_OK;
  OURO_DISPATCH(H->d.variant, return ouro::launch::round_fused<V>(H, d_sizes, n, seed, mode, d_out, d_ptrs, work, s));
}

/* The work slot of an eager round on stream s; null (the round then works in
 * its own zeroed result) for a round that is being captured, and where all
 * slots belong to other streams.  A slot belongs to one stream for the heap's
 * life: the launches of a stream run one after another, so no two launches
 * meet on it, however many are in flight and however long one takes.  Streams
 * are told apart by their ids, which are not used again when a stream is
 * destroyed.  A captured round has no such order: its graph may be replayed
 * beside anything, from any stream.  The entries of the table only ever go
 * from 0 to an id, first free entry first, so a stream never gets two. */
static ouro_status round_work(ouro_heap *H, cudaStream_t s, void **work) {
  *work = nullptr;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  OURO_CUDA(cudaStreamIsCapturing(s, &cap));
  if (cap != cudaStreamCaptureStatusNone) return OURO_OK;
  unsigned long long id = 0;
  OURO_CUDA(cudaStreamGetId(s, &id));
  ++id;   /* 0 marks a free entry */
  for (unsigned k = 0; k < OURO_WORK_SLOTS; ++k) {
    unsigned long long have = __atomic_load_n(&H->work_stream[k], __ATOMIC_RELAXED);
    if (!have && __atomic_compare_exchange_n(&H->work_stream[k], &have, id, false, __ATOMIC_RELAXED, __ATOMIC_RELAXED))
      have = id;
    if (have == id) {
      *work = H->meta + H->off_work + (size_t)k * 128;
      break;
    }
  }
  return OURO_OK;
}
}  // namespace host
}  // namespace ouro

extern "C" ouro_status ouro_round_fused(ouro_heap *H, const uint32_t *d_sizes, size_t n, uint32_t seed, int mode,
                                        ouro_check *d_out, void **d_ptrs, void *stream) {
  if (!H || !d_out || (n && !d_sizes)) return OURO_EINVAL;
  if (mode != 0 && mode != 1) return OURO_EINVAL;
  void *work = nullptr;
  if (n) {
    const ouro_status st = ouro::host::round_work(H, S(stream), &work);
    if (st != OURO_OK) return st;
  }
  return ouro::host::round_fused_on(H, d_sizes, n, seed, mode, d_out, d_ptrs, work, S(stream));
}
#endif
