/*
 * Graph growth: adjacency lists that grow inside kernels through the device
 * allocator (a dynamically partitioned workload of the kind Sec. 1 of
 * arXiv 2504.18211 names: graph algorithms need memory repartitioned
 * while the kernel runs).
 *
 * Vertex v owns a list of uint32 neighbours.  It starts with 4 entries
 * (16 B).  When an append does not fit, the list doubles (malloc 2x, copy,
 * free the old list), one doubling at a time, until it reaches one chunk.
 * Past one chunk, entries go to overflow segments of one chunk each, chained
 * newest first: [next pointer (8 B)][entries].
 *
 * A block groups its 2048 (src, dst) pairs by source in a shared-memory hash
 * table, so that every source of the block is one run, and a warp appends 32
 * runs at once, a lane each.  There is no lock: a run reserves its places at
 * the end of its list with one atomic, and the one run that finds the list
 * full grows it (see vertex).  Every wait is bounded; a run whose wait runs
 * out sets the heap's TIMEOUT bit and is skipped (counted in ctl[2]).
 */
#include "ouro_internal.cuh"
#include "ouro_payload.cuh"
#include "ouro_shard.cuh"

using namespace ouro::detail;

namespace {

/* The tail container of a list is its plain array (ovf == 0) or its newest
 * overflow segment; the containers before it are full.  `end` is the
 * reservation word of the tail: entries reserved in the low half; in the high
 * half the plain array's capacity, or TAIL_SEG | the segment's chunk id, so
 * that a reservation in a segment names the segment itself.
 *   - n entries are reserved by one atomic add of n.  Old count + n <=
 *     capacity: the places are the run's own; it writes them and then adds n
 *     to deg (the commit).
 *   - The one run that crosses the capacity (old count <= capacity < old
 *     count + n) owns the places up to the capacity and the growth.  The word
 *     stays past its capacity until the grower publishes the next container
 *     with one exchange, which also drops the counts of the runs that found
 *     it full: those read the word until it is below its capacity and reserve
 *     again.
 *   - A plain array is copied, and freed, only when all its places are
 *     committed (deg equals the capacity), so a run that holds places in it
 *     can read ptr; a full segment is left as it is, so its growth waits for
 *     nobody. */
struct vertex {
  unsigned long long ptr;   /* plain array */
  unsigned long long ovf;   /* newest overflow segment (0: none) */
  unsigned long long end;   /* reservation word of the tail */
  unsigned long long pad0;
  unsigned deg;             /* entries written */
  unsigned pad1;
};

constexpr unsigned TAIL_SEG = 0x80000000u;   /* capacities (2^18 at most) and chunk ids (2^28) stay below */

constexpr int EDGES_PER_THREAD = 8;
constexpr int GB_THREADS = 256;
constexpr int GB_EDGES = EDGES_PER_THREAD * GB_THREADS;   /* 2048 pairs per block */
constexpr int GB_TABLE = 2 * GB_EDGES;                    /* hash slots: half of them used at most */

template <int V>
__global__ void k_graph_init(ouro_heap_dev h, vertex *vt, unsigned nv, unsigned long long *ctl) {
  for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
    void *p = malloc_v<V>(h, 16);
    vt[v].ptr = reinterpret_cast<unsigned long long>(p);
    vt[v].ovf = 0;
    vt[v].end = pack(p ? 4 : 0, 0);
    vt[v].deg = 0;
    if (!p) atomicAdd(&ctl[1], 1ull);
  }
}

constexpr unsigned LANE_ENTRIES = 8;    /* longer runs are written by the whole warp */
constexpr unsigned LANE_COPY = 32;      /* entries of a list that its grower's lane copies alone */

/* A warp appends up to 32 runs, a lane each (n = 0: no run): the n entries at
 * `from` (shared memory) to vertex vx, no vertex twice in a warp.  The lanes
 * go through the protocol of `vertex` in step, so the allocator is called by
 * the whole warp, for all of its growing lists at once.  One round is a
 * reservation, the writes and their commit, about three dependent L2 round
 * trips; what is left to wait for is looked at once a round.  A warp per run
 * under the vertex's lock took about 5 us for each run and one atomic on the
 * appended count per run: 2^22 edges on 2^18 vertices 5570 us, 660 so (with
 * uniform sources 580: what bounds it is the chain of each warp's 32 runs,
 * about 16 us, and not the largest list).  Adds the lane's
 * entries written, dropped (no memory) and skipped (a wait ran out). */
template <int V>
__device__ void warp_append(const ouro_heap_dev &h, vertex *vx, const unsigned *from, unsigned n, unsigned &written,
                            unsigned &dropped, unsigned &skipped) {
  constexpr unsigned FULL = 0xffffffffu;
  const unsigned lane = laneid();
  const unsigned max_plain = h.chunk_bytes >> 2;          /* entries in one chunk */
  const unsigned seg_cap = (h.chunk_bytes - 8) >> 2;     /* entries per overflow segment */
  enum { RESERVE, WAIT, GROW, DONE };
  int st = n ? RESERVE : DONE;
  unsigned tail = 0;                                      /* GROW: high half of the full tail's word */
  unsigned ns = h.backoff_min_ns;
  auto capacity = [&](unsigned t) { return t & TAIL_SEG ? seg_cap : t; };
  for (unsigned long long it = 0; __any_sync(FULL, st != DONE);) {
    bool progress = false;
    unsigned m = 0, at = 0;                               /* places this round: [at, at + m) of `to` */
    unsigned long long to = 0;
    const bool out_of_time = it >= 4ull * h.spin_limit;   /* naps of at most 256 ns */

    /* 1. growth */
    const unsigned cap = capacity(tail);
    const bool plain = !(tail & TAIL_SEG) && tail && tail < max_plain;
    unsigned long long ptr = 0;
    bool grow = false;
    if (st == GROW) {
      if (plain) ptr = ld_rlx(&vx->ptr);
      grow = !plain || ld_acq32(&vx->deg) == cap;
    }
    if (__any_sync(FULL, grow)) {
      __syncwarp();
      unsigned char *fresh =
          static_cast<unsigned char *>(malloc_v<V>(h, plain ? (size_t)cap * 8 : h.chunk_bytes, grow));
      __syncwarp();
      unsigned long long old = 0;
      const bool ok = grow && fresh;
      if (ok && plain && cap <= LANE_COPY) {
        const uint4 *s4 = reinterpret_cast<const uint4 *>(ptr);
        uint4 *d4 = reinterpret_cast<uint4 *>(fresh);
        uint4 v[LANE_COPY / 4];
#pragma unroll
        for (unsigned i = 0; i < LANE_COPY / 4; ++i)
          if (4 * i < cap) v[i] = __ldcg(s4 + i);
#pragma unroll
        for (unsigned i = 0; i < LANE_COPY / 4; ++i)
          if (4 * i < cap) d4[i] = v[i];
      }
      for (unsigned big = __ballot_sync(FULL, ok && plain && cap > LANE_COPY); big; big &= big - 1) {
        const int j = __ffs(big) - 1;
        const uint4 *s4 = reinterpret_cast<const uint4 *>(__shfl_sync(FULL, ptr, j));
        uint4 *d4 = reinterpret_cast<uint4 *>(__shfl_sync(FULL, reinterpret_cast<unsigned long long>(fresh), j));
        const unsigned c4 = __shfl_sync(FULL, cap, j) >> 2;
#pragma unroll 4
        for (unsigned i = lane; i < c4; i += 32) d4[i] = __ldcg(s4 + i);
      }
      unsigned next = 0;
      if (ok) {
        if (plain) {
          old = ptr;
          next = 2 * cap;
          at = cap;
          to = reinterpret_cast<unsigned long long>(fresh);
          vx->ptr = to;
        } else {
          *reinterpret_cast<unsigned long long *>(fresh) =
              tail & TAIL_SEG ? reinterpret_cast<unsigned long long>(seg_of(h, tail & ~TAIL_SEG)) : 0;
          next = TAIL_SEG | (unsigned)((fresh - h.base) >> h.log2_chunk);
          to = reinterpret_cast<unsigned long long>(fresh) + 8;
          vx->ovf = reinterpret_cast<unsigned long long>(fresh);
        }
        m = min(n, capacity(next) - at);
      }
      __threadfence();
      __syncwarp();
      if (ok && n == m) {                /* room for all of the run: the others may go on */
        atomicExch(&vx->end, pack(next, at + m));
        st = DONE;
      } else if (ok) {                   /* the new tail is full too: grow on */
        tail = next;
      } else if (grow) {                 /* no memory: the run is dropped, the next one tries again */
        dropped += n;
        atomicExch(&vx->end, pack(tail, cap));
        st = DONE;
      }
      progress |= grow;
      __syncwarp();
      free_v<V>(h, reinterpret_cast<void *>(old));
      __syncwarp();
    }

    /* 2. reservations */
    if (st == WAIT) {
      const unsigned long long e = ld_rlx(&vx->end);
      if (lo32(e) <= capacity(hi32(e))) st = RESERVE;
    }
    if (st == RESERVE) {
      const unsigned long long e = atomicAdd(&vx->end, (unsigned long long)n);
      const unsigned cnt = lo32(e), room = capacity(hi32(e));
      if (cnt <= room) {
        tail = hi32(e);
        m = min(n, room - cnt);
        at = cnt;
        st = m == n ? DONE : GROW;
        fence_acq_rel();
        if (m)
          to = tail & TAIL_SEG ? reinterpret_cast<unsigned long long>(seg_of(h, tail & ~TAIL_SEG)) + 8
                               : ld_rlx(&vx->ptr);
        progress = true;
      } else {
        st = WAIT;
      }
    }

    /* 3. writes and commits */
    if (__any_sync(FULL, m)) {
      unsigned *dst = reinterpret_cast<unsigned *>(to) + at;
      if (m <= LANE_ENTRIES)
        for (unsigned i = 0; i < m; ++i) dst[i] = from[i];
      for (unsigned big = __ballot_sync(FULL, m > LANE_ENTRIES); big; big &= big - 1) {
        const int j = __ffs(big) - 1;
        unsigned *d = reinterpret_cast<unsigned *>(__shfl_sync(FULL, reinterpret_cast<unsigned long long>(dst), j));
        const unsigned *f =
            reinterpret_cast<const unsigned *>(__shfl_sync(FULL, reinterpret_cast<unsigned long long>(from), j));
        const unsigned k = __shfl_sync(FULL, m, j);
        for (unsigned i = lane; i < k; i += 32) d[i] = f[i];
      }
      __threadfence();
      __syncwarp();
      if (m) {
        atomicAdd(&vx->deg, m);
        written += m;
        from += m;
        n -= m;
      }
    }

    /* 4. nothing moved: back off; give up when the wait runs out */
    if (__any_sync(FULL, progress)) {
      ns = h.backoff_min_ns;
      continue;
    }
    if (out_of_time) {
      if (st != DONE) {
        set_error(h, OURO_ERR_TIMEOUT, OURO_SITE_GRAPH_LOCK);
        skipped += n;
        if (st == GROW) atomicExch(&vx->end, pack(tail, capacity(tail)));
        st = DONE;
      }
      continue;
    }
    ++it;
    __nanosleep(ns);
    ns = min(ns * 2, 256u);
  }
}

/* Groups the block's pairs by source and appends one run per source.  The
 * grouping only needs equal sources together, so a hash table takes the place
 * of a sort: an edge finds its source's slot (linear probing) and its rank
 * among the slot's edges with shared-memory atomics, a scan over the slots
 * gives every run its place in `sorted`.  (The bitonic sort of 4096 64-bit
 * keys that it replaces took 78 passes over shared memory.) */
template <int V>
__global__ void __launch_bounds__(GB_THREADS, ouro_page_queues(V) ? 3 : 2)
k_graph_insert(ouro_heap_dev h, vertex *vt, const unsigned *src, const unsigned *dst, unsigned long long n_edges,
               unsigned long long *ctl) {
  __shared__ unsigned key[GB_TABLE];                  /* source + 1 (0: free) */
  __shared__ unsigned cnt[GB_TABLE];                  /* edges of the slot, then the end of its run */
  __shared__ unsigned sorted[GB_EDGES];
  __shared__ unsigned short run_slot[GB_EDGES];       /* slots in use, in slot order */
  __shared__ unsigned warp_sum[GB_THREADS / 32];
  __shared__ unsigned sums[3];                        /* written, dropped, skipped */
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long base = (unsigned long long)blockIdx.x * GB_EDGES;
  for (unsigned i = threadIdx.x; i < GB_TABLE; i += GB_THREADS) key[i] = cnt[i] = 0;
  if (threadIdx.x < 3) sums[threadIdx.x] = 0;
  unsigned s[EDGES_PER_THREAD], d[EDGES_PER_THREAD];
#pragma unroll
  for (int k = 0; k < EDGES_PER_THREAD; ++k) {
    const unsigned long long e = base + k * GB_THREADS + threadIdx.x;
    s[k] = e < n_edges ? src[e] + 1 : 0;
    d[k] = e < n_edges ? dst[e] : 0;
  }
  __syncthreads();
  unsigned place[EDGES_PER_THREAD];                   /* rank << 16 | slot */
#pragma unroll
  for (int k = 0; k < EDGES_PER_THREAD; ++k) {
    if (!s[k]) continue;
    unsigned slot_i = (s[k] * 0x9E3779B1u) >> 20;     /* 12 bits: GB_TABLE slots */
    for (;;) {                                        /* ends: half of the slots stay free */
      const unsigned seen = key[slot_i] == s[k] ? s[k] : atomicCAS(&key[slot_i], 0u, s[k]);
      if (seen == 0 || seen == s[k]) break;
      slot_i = (slot_i + 1) & (GB_TABLE - 1);
    }
    place[k] = atomicAdd(&cnt[slot_i], 1u) << 16 | slot_i;
  }
  __syncthreads();
  /* scan: edges (high half) and slots in use (low half) before each slot */
  constexpr unsigned PER = GB_TABLE / GB_THREADS;
  unsigned mine = 0;
#pragma unroll
  for (unsigned k = 0; k < PER; ++k) {
    const unsigned c = cnt[threadIdx.x * PER + k];
    mine += c << 16 | (c != 0);
  }
  unsigned incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
    if ((int)lane >= o) incl += y;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  unsigned before = incl - mine, n_runs = 0;
#pragma unroll
  for (unsigned w = 0; w < GB_THREADS / 32; ++w) {
    if (w < warp) before += warp_sum[w];
    n_runs += warp_sum[w] & 0xFFFFu;
  }
#pragma unroll
  for (unsigned k = 0; k < PER; ++k) {
    const unsigned i = threadIdx.x * PER + k, c = cnt[i];
    if (c) run_slot[before & 0xFFFFu] = (unsigned short)i;
    before += c << 16 | (c != 0);
    cnt[i] = (before >> 16) << 16 | c;                /* end of the run << 16 | its length */
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < EDGES_PER_THREAD; ++k) {
    if (!s[k]) continue;
    const unsigned c = cnt[place[k] & 0xFFFFu];
    sorted[(c >> 16) - (c & 0xFFFFu) + (place[k] >> 16)] = d[k];
  }
  __syncthreads();
  unsigned written = 0, dropped = 0, skipped = 0;
  for (unsigned r0 = warp * 32; r0 < n_runs; r0 += GB_THREADS) {
    const unsigned r = r0 + lane;
    const unsigned i = r < n_runs ? run_slot[r] : 0, c = r < n_runs ? cnt[i] : 0, n = c & 0xFFFFu;
    warp_append<V>(h, vt + (n ? key[i] - 1 : 0), sorted + ((c >> 16) - n), n, written, dropped, skipped);
  }
  written = __reduce_add_sync(0xffffffffu, written);
  dropped = __reduce_add_sync(0xffffffffu, dropped);
  skipped = __reduce_add_sync(0xffffffffu, skipped);
  if (lane == 0) {
    if (written) atomicAdd(&sums[0], written);
    if (dropped) atomicAdd(&sums[1], dropped);
    if (skipped) atomicAdd(&sums[2], skipped);
  }
  __syncthreads();
  if (threadIdx.x < 3 && sums[threadIdx.x]) atomicAdd(&ctl[threadIdx.x], (unsigned long long)sums[threadIdx.x]);
}

/* Every vertex's entries, plain array then overflow segments (newest first),
 * into out[off[v] .. off[v] + deg[v]).  A warp copies the plain array of one
 * vertex; the block's vertices with segments follow one by one, all threads
 * copying a segment while its link is read.  The chain of links bounds it: 86
 * of them for a list of 175,000 entries, which one warp alone copied in 1.3
 * ms (2^22 entries of 2^18 vertices: 1380 us so, 270 with the block, and less
 * with its loads in flight past the ragged end of a segment, whose remainder
 * loop had cost two of its threads seven round trips a segment). */
__global__ void __launch_bounds__(256) k_graph_gather(const vertex *vt, unsigned nv, const unsigned long long *off,
                                                      unsigned *out, unsigned chunk_bytes) {
  constexpr unsigned WARPS = 8;
  __shared__ unsigned long long s_seg[WARPS], s_out[WARPS];
  __shared__ unsigned s_take[WARPS];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned max_plain = chunk_bytes >> 2, seg_cap = (chunk_bytes - 8) >> 2;
  for (unsigned long long v0 = (unsigned long long)blockIdx.x * WARPS; v0 < nv;
       v0 += (unsigned long long)gridDim.x * WARPS) {
    const unsigned long long v = v0 + warp;
    unsigned long long seg = 0;
    if (v < nv) {
      unsigned long long o = off[v];
      const vertex x = vt[v];
      const unsigned *pl = reinterpret_cast<const unsigned *>(x.ptr);
      const unsigned cnt = x.ovf ? (x.ptr ? max_plain : 0) : lo32(x.end);
#pragma unroll 4
      for (unsigned i = lane; i < cnt; i += 32) out[o + i] = pl[i];
      seg = x.ovf;
      if (lane == 0) {
        s_out[warp] = o + cnt;
        s_take[warp] = lo32(x.end);
      }
    }
    if (lane == 0) s_seg[warp] = seg;
    if (!__syncthreads_or(seg != 0)) continue;
    for (unsigned w = 0; w < WARPS; ++w) {
      unsigned long long sg = s_seg[w], o = s_out[w];
      unsigned take = s_take[w];
      for (unsigned k = 0; sg && k < (1u << 26); ++k) {
        const unsigned long long next = *reinterpret_cast<const unsigned long long *>(sg);
        const unsigned *e = reinterpret_cast<const unsigned *>(sg + 8);
        for (unsigned i0 = threadIdx.x; i0 < take; i0 += 8 * 256) {   /* eight loads in flight, the ragged end too */
          unsigned d[8];
#pragma unroll
          for (unsigned j = 0; j < 8; ++j)
            if (i0 + 256 * j < take) d[j] = e[i0 + 256 * j];
#pragma unroll
          for (unsigned j = 0; j < 8; ++j)
            if (i0 + 256 * j < take) out[o + i0 + 256 * j] = d[j];
        }
        o += take;
        sg = next;
        take = seg_cap;
      }
    }
    __syncthreads();
  }
}

/* Frees every list.  A lane per vertex; a segment's link is read before the
 * frees of the segment before it wait for their queue slots.  The classes are
 * in the records too, but the frees look every block up in the chunk table: a
 * table from before a reset of the heap, or of another heap, records bad frees
 * and leaves the queues alone. */
template <int V>
__global__ void k_graph_free(ouro_heap_dev h, vertex *vt, unsigned nv) {
  const unsigned threads = gridDim.x * blockDim.x;
  for (unsigned v0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); v0 < nv; v0 += threads) {
    const unsigned v = v0 + (threadIdx.x & 31);
    unsigned long long ptr = 0, seg = 0;
    if (v < nv) {
      ptr = vt[v].ptr;
      seg = vt[v].ovf;
    }
    unsigned long long next = seg ? *reinterpret_cast<const unsigned long long *>(seg) : 0;
    __syncwarp();
    free_v<V>(h, reinterpret_cast<void *>(ptr));
    for (unsigned guard = 0; __any_sync(0xffffffffu, seg != 0) && guard < (1u << 26); ++guard) {
      const unsigned long long after = next ? *reinterpret_cast<const unsigned long long *>(next) : 0;
      __syncwarp();
      free_v<V>(h, reinterpret_cast<void *>(seg));
      __syncwarp();
      seg = next;
      next = after;
    }
    if (v < nv) vt[v].ptr = vt[v].ovf = 0;
  }
}

#if OURO_SHARD_ENTRIES
inline cudaStream_t S(void *s) { return reinterpret_cast<cudaStream_t>(s); }
#endif

}  // namespace

/* ------------------------------------------------------- per-form launchers */
namespace ouro {
namespace launch {

template <int V>
ouro_status graph_init(ouro_heap *H, void *d_vertices, uint32_t n_vertices, unsigned long long *d_ctl,
                       cudaStream_t s) {
  k_graph_init<V><<<4 * ouro::host::sm_count(), 256, 0, s>>>(H->d, (vertex *)d_vertices, n_vertices, d_ctl);
  OURO_LAUNCHED();
  return OURO_OK;
}

template <int V>
ouro_status graph_insert(ouro_heap *H, void *d_vertices, const uint32_t *d_src, const uint32_t *d_dst,
                         uint64_t n_edges, unsigned long long *d_ctl, cudaStream_t s) {
  const unsigned blocks = (unsigned)((n_edges + GB_EDGES - 1) / GB_EDGES);
  k_graph_insert<V><<<blocks, GB_THREADS, 0, s>>>(H->d, (vertex *)d_vertices, d_src, d_dst, n_edges, d_ctl);
  OURO_LAUNCHED();
  return OURO_OK;
}

template <int V>
ouro_status graph_free(ouro_heap *H, void *d_vertices, uint32_t n_vertices, cudaStream_t s) {
  k_graph_free<V><<<4 * ouro::host::sm_count(), 256, 0, s>>>(H->d, (vertex *)d_vertices, n_vertices);
  OURO_LAUNCHED();
  return OURO_OK;
}

#define INST_GRAPH_INIT(PRE, V) \
  PRE template ouro_status graph_init<V>(ouro_heap *, void *, uint32_t, unsigned long long *, cudaStream_t);
#define INST_GRAPH_INSERT(PRE, V)                                                                          \
  PRE template ouro_status graph_insert<V>(ouro_heap *, void *, const uint32_t *, const uint32_t *, uint64_t, \
                                           unsigned long long *, cudaStream_t);
#define INST_GRAPH_FREE(PRE, V) PRE template ouro_status graph_free<V>(ouro_heap *, void *, uint32_t, cudaStream_t);
OURO_SHARD_INSTANTIATE(INST_GRAPH_INIT)
OURO_SHARD_INSTANTIATE(INST_GRAPH_INSERT)
OURO_SHARD_INSTANTIATE(INST_GRAPH_FREE)

}  // namespace launch
}  // namespace ouro

#if OURO_SHARD_ENTRIES
extern "C" size_t ouro_graph_vertex_bytes(void) { return sizeof(vertex); }

extern "C" ouro_status ouro_graph_init(ouro_heap *H, void *d_vertices, uint32_t n_vertices, unsigned long long *d_ctl,
                                       void *stream) {
  if (!H || !d_vertices || !d_ctl || !n_vertices) return OURO_EINVAL;
  OURO_CUDA(cudaMemsetAsync(d_ctl, 0, 4 * 8, S(stream)));
  OURO_DISPATCH(H->d.variant, return ouro::launch::graph_init<V>(H, d_vertices, n_vertices, d_ctl, S(stream)));
}

extern "C" ouro_status ouro_graph_insert(ouro_heap *H, void *d_vertices, const uint32_t *d_src, const uint32_t *d_dst,
                                         uint64_t n_edges, unsigned long long *d_ctl, void *stream) {
  if (!H || !d_vertices || !d_ctl || (n_edges && (!d_src || !d_dst))) return OURO_EINVAL;
  if (!n_edges) return OURO_OK;
  OURO_DISPATCH(H->d.variant,
                return ouro::launch::graph_insert<V>(H, d_vertices, d_src, d_dst, n_edges, d_ctl, S(stream)));
}

extern "C" ouro_status ouro_graph_gather(ouro_heap *H, const void *d_vertices, uint32_t n_vertices,
                                         const unsigned long long *d_offsets, uint32_t *d_out, void *stream) {
  if (!H || !d_vertices || !d_offsets || !d_out) return OURO_EINVAL;
  const int g = 8 * ouro::host::sm_count();
  k_graph_gather<<<g, 256, 0, S(stream)>>>((const vertex *)d_vertices, n_vertices, d_offsets, d_out, H->d.chunk_bytes);
  OURO_LAUNCHED();
  return OURO_OK;
}

extern "C" ouro_status ouro_graph_free(ouro_heap *H, void *d_vertices, uint32_t n_vertices, void *stream) {
  if (!H || !d_vertices) return OURO_EINVAL;
  OURO_DISPATCH(H->d.variant, return ouro::launch::graph_free<V>(H, d_vertices, n_vertices, S(stream)));
}
#endif
