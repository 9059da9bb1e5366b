/* Device helpers shared by the library's kernels: variant-resolved
 * malloc / free, and the warp-cooperative driver-round payload (Sec. 3 of
 * arXiv 2504.18211: write data into each block, read it back, check it). */
#ifndef OURO_PAYLOAD_CUH
#define OURO_PAYLOAD_CUH

#include "ouro_internal.cuh"

namespace ouro {
namespace detail {


/* Variant-resolved malloc.  want = false: the lane asks for nothing but
 * stays in the call to help its warp carve (see page_malloc).  FILL: slot
 * writes in flight per lane when the warp fills a carve (page queues). */
template <int V, int FILL = 1>
__device__ __forceinline__ void *malloc_v(const ouro_heap_dev &h, unsigned long long n, bool want = true) {
  const unsigned mask = __activemask();
  const int cls = want ? size_class(h, n) : -1;
  if (want && cls < 0) stat_add(h, OURO_ROW_NONE, n == 0 ? OURO_ST_ZERO : OURO_ST_TOO_LARGE, 1);
  if (!__any_sync(mask, cls >= 0)) return nullptr;
  if constexpr (ouro_page_queues(V)) return page_malloc<V, FILL>(h, cls, mask);   /* pages and runs */
  else return chunk_or_run_malloc<V>(h, cls, mask);
}

/* Class and item of a block being freed; -1 for null or an invalid free
 * (recorded).  A run is marked free here; page queues in checked mode clear
 * the page's bit and catch a double free. */
template <int V>
__device__ __forceinline__ int free_locate(const ouro_heap_dev &h, void *p, unsigned &item) {
  int cls = -1;
  if (p) {
    cls = locate(h, p, &item);
    if (cls < 0) set_error(h, OURO_ERR_BAD_FREE, OURO_SITE_BAD_FREE);
    else if (cls >= (int)h.n_classes) {   /* a run */
      if (!run_mark_free(h, cls, item)) cls = -1;
    } else if (h.checked && ouro_page_queues(V)) {
      const unsigned sh = h.log2_chunk - 4 - cls;
      const unsigned pg = item & ((1u << sh) - 1), x = item >> sh, bit = 1u << (pg & 31);
      __threadfence();
      unsigned old = atomicOr(&h.bits[(size_t)x * h.words_per_chunk + (pg >> 5)], bit);
      if (old & bit) {
        set_error(h, OURO_ERR_DOUBLE_FREE, OURO_SITE_PAGE_DOUBLE);
        cls = -1;
      }
    }
  }
  return cls;
}

/* FENCE = false: only for kernels that free blocks written before they began
 * and allocate nothing (the batch free kernel).  known_cls >= 0: the caller
 * allocated p itself with that class; a page's chunk-table lookup (one L2
 * round trip) is then left out, as in stage_free. */
template <int V, bool FENCE = true>
__device__ __forceinline__ void free_v(const ouro_heap_dev &h, void *p, int known_cls = -1) {
  const unsigned mask = __activemask();
  unsigned item = 0;
  int cls;
  if (p && known_cls >= 0 && known_cls < (int)h.n_classes && !(ouro_page_queues(V) && h.checked)) {
    cls = known_cls;
    item = (unsigned)(((const unsigned char *)p - h.base) >> (4 + cls));
  } else {
    cls = free_locate<V>(h, p, item);
  }
  if constexpr (!ouro_page_queues(V)) {
    chunk_or_run_free<V, FENCE>(h, cls, item, p, mask);
  } else {
    const unsigned vmask = __ballot_sync(mask, cls >= 0);
    if (cls < 0) return;
    page_free<V>(h, cls, item, vmask);
  }
}

/* Staged malloc: the warp's shared-memory stacks first (every queue form), then
 * the heap. */
template <int V, int WARPS>
__device__ __forceinline__ void *stage_malloc_v(ouro_block_ctx<WARPS> &ctx, const ouro_heap_dev &h,
                                                unsigned long long n, bool want) {
  return ouro::detail::stage_malloc<V, WARPS>(ctx, h, n, want);
}

/* ------------------------------------------------------------- payload */
/* MurmurHash3 32-bit finalizer (Appleby, public domain) */
__device__ __forceinline__ uint32_t fmix32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x85ebca6bu;
  x ^= x >> 13;
  x *= 0xc2b2ae35u;
  x ^= x >> 16;
  return x;
}
#define OURO_GOLD 0x9E3779B9u

/* per-lane check counters: mismatches and the XOR fold in 32 bits (the
 * words are 32-bit), the sum and the word count in 64 */
struct payload_acc {
  unsigned mism = 0, x = 0;
  unsigned long long s = 0, words = 0;
  __device__ void fold(uint32_t v) {
    x ^= v;
    s += v;
  }
};

/* Warp-cooperative payload over the blocks held by the lanes of a warp (every
 * lane calls; a lane without a block passes p = null).
 *   WRITE:  store the pattern.
 *   CHECK:  read back, compare, fold the checksums into a.
 *   FUSED:  write, then (after __syncwarp) read back through L2 with every
 *           lane checking what a neighbour wrote.
 * mode 0: word 0 = tid.  mode 1: floor(size/4) words key + w*GOLD, then the
 * low size%4 bytes of word floor(size/4).
 *
 * A block is cut into 16-byte units and a rest of up to 15 bytes.  What
 * bounds the payload of small blocks is the chain of L2 round trips, so the
 * blocks of up to pay_flat units are laid end to end and the 32 lanes stride
 * over the whole row of units, four loads in flight per lane: a row of 32
 * blocks of 16 B is one store and one load per lane instead of 32 round
 * trips with 31 lanes idle (3 * 2^18 blocks of 64 B: write 45 -> 17 us, check
 * 88 -> 20 us; a fused round of 10,240 blocks of 16 B 37 -> 12 us, 11 since).  Larger
 * blocks fill the warp by themselves and go one at a time, so that a block is
 * read back while L2 still holds it (laying all 32 end to end pushed most of
 * the read-back out to DRAM).  The rests are done by the lanes that hold the
 * blocks, all at once, instead of by one lane block after block. */
enum { PAY_WRITE = 1, PAY_CHECK = 2, PAY_FUSED = 3 };
/* units of the largest block that goes into the row: where the row writes and
 * reads back, its longer stretch between the two costs a little on a full
 * chip (2^20 sweep: 16 units 315 us, 32 units 317, 64 units 326), so it stays
 * shorter than where a kernel does one of the two */
__host__ __device__ constexpr unsigned pay_flat(int op) { return op == PAY_FUSED ? 16u : 64u; }

__device__ __forceinline__ uint4 pat4(uint32_t v) {
  return make_uint4(v, v + OURO_GOLD, v + 2u * OURO_GOLD, v + 3u * OURO_GOLD);
}
__device__ __forceinline__ uint4 pat4(uint32_t key, uint32_t w0) { return pat4(key + w0 * OURO_GOLD); }

__device__ __forceinline__ void check4(const uint4 &got, const uint4 &want, payload_acc &a) {
  a.mism += (got.x != want.x) + (got.y != want.y) + (got.z != want.z) + (got.w != want.w);
  a.x ^= got.x ^ got.y ^ got.z ^ got.w;
  a.s += (unsigned long long)got.x + got.y + got.z + got.w;
}

/* Payload units pass through L2 once, so stores and loads carry the
 * evict_first policy: a unit that was read back is the next to leave L2, and
 * the dirty lines go out to HBM about in the order they were written, instead
 * of in the order of an LRU over all of L2 (which also held the allocator's
 * slots and tables).  2^20 fused size-sweep round: 326 -> 315 us; the policy
 * on the stores alone 351 us (the read-back renewed the lines), on the loads
 * alone 330.  ld.global.cg reads L2, past any line of L1. */
__device__ __forceinline__ unsigned long long stream_policy(bool plain = false) {
  unsigned long long pol;
  if (plain) asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  else asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void st_stream(uint4 *p, const uint4 &v, unsigned long long pol) {
  asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w), "l"(pol)
               : "memory");
}
__device__ __forceinline__ uint4 ld_stream(const uint4 *p, unsigned long long pol) {
  uint4 v;
  asm volatile("ld.global.cg.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol) : "memory");
  return v;
}

/* the words past the last whole unit and the tail bytes of one block, by one
 * lane; the loads of the read-back are independent of each other */
template <bool WRITE>
__device__ __forceinline__ void block_rest(unsigned char *bp, uint32_t key, uint32_t size, payload_acc &a) {
  const uint32_t nw = size >> 2, tail = size & 3, w0 = nw & ~3u, k = nw & 3u;
  uint32_t *wp = reinterpret_cast<uint32_t *>(bp) + w0;
  unsigned char *tb = bp + 4ull * nw;
  const uint32_t v = key + nw * OURO_GOLD;
  if (WRITE) {
#pragma unroll
    for (uint32_t w = 0; w < 3; ++w)
      if (w < k) wp[w] = key + (w0 + w) * OURO_GOLD;
#pragma unroll
    for (uint32_t b = 0; b < 3; ++b)
      if (b < tail) tb[b] = (unsigned char)(v >> (8 * b));
  } else {
    uint32_t g[3], t[3];
#pragma unroll
    for (uint32_t w = 0; w < 3; ++w) g[w] = w < k ? __ldcg(wp + w) : 0u;
#pragma unroll
    for (uint32_t b = 0; b < 3; ++b) t[b] = b < tail ? __ldcg(tb + b) : 0u;
#pragma unroll
    for (uint32_t w = 0; w < 3; ++w) {
      a.mism += w < k && g[w] != key + (w0 + w) * OURO_GOLD;
      a.fold(g[w]);
    }
#pragma unroll
    for (uint32_t b = 0; b < 3; ++b) a.mism += b < tail && t[b] != ((v >> (8 * b)) & 0xFFu);
    a.fold(t[0] | t[1] << 8 | t[2] << 16);
  }
}

/* Lane whose block holds unit f of the row: the number of lanes whose
 * running count incl does not pass f (31 at most). */
__device__ __forceinline__ unsigned row_owner(unsigned incl, unsigned f) {
  unsigned j = 0;
#pragma unroll
  for (unsigned s = 16; s; s >>= 1)
    if (__shfl_sync(0xffffffffu, incl, j + s - 1) <= f) j += s;
  return j;
}

/* The row of small blocks (n_units > 0 for a lane whose block is in it) and
 * every block's rest.  Out of line: its registers (four loads in flight and
 * their places in the row) stay out of the allocating kernels' budget. */
template <int OP, bool PLAIN>
__device__ __noinline__ payload_acc payload_row(unsigned char *p, uint32_t size, uint32_t key, uint32_t n_units,
                                                bool plain = false) {
  constexpr unsigned FULL = 0xffffffffu;
  const unsigned lane = laneid();
  const unsigned rd = OP == PAY_FUSED ? (lane + 1) & 31 : lane;   /* lane whose units this lane checks */
  const unsigned long long pol = stream_policy(PLAIN && plain);
  payload_acc a;
  uint32_t incl = n_units;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, incl, o);
    if ((int)lane >= o) incl += y;
  }
  const uint32_t total = __shfl_sync(FULL, incl, 31);
  const uint32_t excl = incl - n_units;
  /* unit f of the row, in this lane's block: address row_p + 16 f, first word row_k + 4 f * GOLD */
  const unsigned long long row_p = reinterpret_cast<unsigned long long>(p) - 16ull * excl;
  const uint32_t row_k = key - 4u * excl * OURO_GOLD;
  if (OP & PAY_WRITE) {
    for (uint32_t f0 = 0; f0 < total; f0 += 32) {
      const uint32_t f = f0 + lane;
      const unsigned j = row_owner(incl, f);
      const unsigned long long bp = __shfl_sync(FULL, row_p, j);
      const uint32_t v = __shfl_sync(FULL, row_k, j);
      if (f < total) st_stream(reinterpret_cast<uint4 *>(bp + 16ull * f), pat4(v, 4 * f), pol);
    }
    if (size & 15) block_rest<true>(p, key, size, a);
  }
  if (OP == PAY_FUSED) __syncwarp();
  if (OP & PAY_CHECK) {
    for (uint32_t f0 = 0; f0 < total; f0 += 128) {
      uint4 g[4];
      uint32_t v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t f = f0 + 32 * k + rd;
        const unsigned j = row_owner(incl, f);
        const unsigned long long bp = __shfl_sync(FULL, row_p, j);
        v[k] = __shfl_sync(FULL, row_k, j) + 4 * f * OURO_GOLD;
        if (f < total) g[k] = ld_stream(reinterpret_cast<const uint4 *>(bp + 16ull * f), pol);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (f0 + 32 * k + rd < total) check4(g[k], pat4(v[k]), a);
    }
    if (OP == PAY_FUSED) {
      const unsigned long long np = __shfl_sync(FULL, reinterpret_cast<unsigned long long>(p), rd);
      const uint32_t ns = __shfl_sync(FULL, size, rd), nk = __shfl_sync(FULL, key, rd);
      if (ns & 15) block_rest<false>(reinterpret_cast<unsigned char *>(np), nk, ns, a);
    } else if (size & 15) {
      block_rest<false>(p, key, size, a);
    }
  }
  return a;
}

/* The blocks one after another, each written and read back through L2 before
 * the next (OP as above, FUSED only).  Virtualized lists: a warp that holds
 * its small blocks for the few microseconds of a row takes and gives back
 * queue positions faster than the list's segments, retired in order, come
 * round again, and the queue then holds most of the pages and with them most
 * of the segments (fused rounds of 2^20 requests of 64 B 1290 us, 212 so). */
__device__ __noinline__ inline payload_acc payload_paced(unsigned char *p, uint32_t size, uint32_t key) {
  constexpr unsigned FULL = 0xffffffffu;
  const unsigned lane = laneid(), rd = (lane + 1) & 31;
  payload_acc a;
  for (unsigned todo = __ballot_sync(FULL, size); todo; todo &= todo - 1) {
    const int j = __ffs(todo) - 1;
    unsigned char *bp = reinterpret_cast<unsigned char *>(__shfl_sync(FULL, reinterpret_cast<unsigned long long>(p), j));
    const uint32_t bs = __shfl_sync(FULL, size, j), bkey = __shfl_sync(FULL, key, j), bu = bs >> 4;
    uint4 *u4 = reinterpret_cast<uint4 *>(bp);
    for (uint32_t u = lane; u < bu; u += 32) u4[u] = pat4(bkey, 4 * u);
    if (lane == (bu & 31) && (bs & 15)) block_rest<true>(bp, bkey, bs, a);
    __syncwarp();
    for (uint32_t u = rd; u < bu; u += 32) check4(__ldcg(u4 + u), pat4(bkey, 4 * u), a);
    if (rd == (bu & 31) && (bs & 15)) block_rest<false>(bp, bkey, bs, a);
  }
  return a;
}

/* Mean payload units of a task's blocks up to which they are paced, on lists of
 * pages: 24 unstaged (2^20 requests of 256 B: 193 to 1380 us from run to run,
 * paced 216; of 384 B 230 to 990, paced 227; any size up to 600 B 290, and up to
 * 1300 where the host waits for every round, paced 350), 8 staged (64 B: 266 to
 * 1290, paced 222; 256 B 188, paced 227). */
__host__ __device__ constexpr unsigned pace_payload(int v, bool stage) {
  return v != OURO_PAGE_VLIST ? 0u : stage ? 8u : 24u;
}

/* Unstaged rounds on plain page arrays: pages come and go in queue order, so a
 * page is not seen again before all others, and in a large batch neither the
 * evict_first policy nor a row that holds less than a sixteenth of its task's
 * units pays.  2^20 size sweep: 380 us with both, 371 without the policy, 363
 * without either; a row of all blocks of 64 B 97 and 95 us, any size up to 600
 * B 197 and 183.  10,240 blocks of 16 B: 14.8 us with the policy, 15.4 without.
 * (On virtualized queues the policy is worth more than in staged rounds: 422 us
 * with it on a list and 490 without, 340 and 424 on an array.) */
__host__ __device__ constexpr bool plain_payload(int v, bool stage) { return v == OURO_PAGE_ARRAY && !stage; }
constexpr uint32_t PAY_PLAIN_SHARE = 16;

/* PLAIN: see plain_payload; PACE: see pace_payload (0: not).  Both only where
 * the warp's tasks have 16 requests or more (wide), as in every large batch. */
template <int OP, bool PLAIN = false, unsigned PACE = 0>
__device__ __forceinline__ void warp_payload(unsigned char *p, uint32_t size, uint32_t tid, uint32_t seed, int mode,
                                             payload_acc &a, bool wide = false) {
  constexpr unsigned FULL = 0xffffffffu;
  const unsigned lane = laneid();
  if (mode == 0) {
    if (p) {
      if (OP & PAY_WRITE) *reinterpret_cast<uint32_t *>(p) = tid;
      if (OP == PAY_FUSED) __syncwarp(__activemask());
      if (OP & PAY_CHECK) {
        uint32_t v = __ldcg(reinterpret_cast<const uint32_t *>(p));
        a.mism += v != tid;
        a.fold(v);
        a.words++;
      }
    }
    return;
  }
  const uint32_t key = fmix32(seed ^ (tid * OURO_GOLD));
  if (!p) size = 0;
  const unsigned rd = OP == PAY_FUSED ? (lane + 1) & 31 : lane;   /* lane whose units this lane checks */
  const uint32_t units = size >> 4;
  bool flat = units <= pay_flat(OP);
  if (PLAIN && OP == PAY_FUSED && wide) {
    const uint32_t row = __reduce_add_sync(FULL, flat ? units : 0u), rest = __reduce_add_sync(FULL, flat ? 0u : units);
    if (rest > PAY_PLAIN_SHARE * row) flat = units == 0;
  }
  if (OP & PAY_CHECK) a.words += (size >> 2) + ((size & 3) != 0);
  if (OP == PAY_FUSED && PACE && wide &&
      __reduce_add_sync(FULL, units < 32u * PACE ? units : 32u * PACE) < PACE * __popc(__ballot_sync(FULL, size != 0)) + 1) {
    const payload_acc r = payload_paced(p, size, key);
    a.mism += r.mism;
    a.x ^= r.x;
    a.s += r.s;
    return;
  }
  if (__any_sync(FULL, (flat && units) || (size & 15))) {
    const payload_acc r = payload_row<OP, PLAIN>(p, size, key, flat ? units : 0, wide);
    a.mism += r.mism;
    a.x ^= r.x;
    a.s += r.s;
  }

  /* the larger blocks, one at a time */
  unsigned big = __ballot_sync(FULL, !flat);
  if (!big) return;
  const unsigned long long pol = stream_policy(PLAIN && wide);
  for (; big; big &= big - 1) {
    const int j = __ffs(big) - 1;
    uint4 *u4 = reinterpret_cast<uint4 *>(__shfl_sync(FULL, reinterpret_cast<unsigned long long>(p), j));
    const uint32_t bu = __shfl_sync(FULL, units, j), bkey = __shfl_sync(FULL, key, j);
    if (OP & PAY_WRITE) {
#pragma unroll 4
      for (uint32_t u = lane; u < bu; u += 32) st_stream(u4 + u, pat4(bkey, 4 * u), pol);
    }
    if (OP == PAY_FUSED) __syncwarp();
    if (OP & PAY_CHECK) {
      uint32_t u = rd;
      for (; u + 96 < bu; u += 128) {          /* four independent 16-byte loads in flight */
        const uint4 g0 = ld_stream(u4 + u, pol), g1 = ld_stream(u4 + u + 32, pol), g2 = ld_stream(u4 + u + 64, pol),
                    g3 = ld_stream(u4 + u + 96, pol);
        check4(g0, pat4(bkey, 4 * u), a);
        check4(g1, pat4(bkey, 4 * (u + 32)), a);
        check4(g2, pat4(bkey, 4 * (u + 64)), a);
        check4(g3, pat4(bkey, 4 * (u + 96)), a);
      }
      if (u + 32 < bu) {
        const uint4 g0 = ld_stream(u4 + u, pol), g1 = ld_stream(u4 + u + 32, pol);
        check4(g0, pat4(bkey, 4 * u), a);
        check4(g1, pat4(bkey, 4 * (u + 32)), a);
        u += 64;
      }
      if (u < bu) check4(ld_stream(u4 + u, pol), pat4(bkey, 4 * u), a);
    }
  }
}

/* block reduction of the check counters into sm (shared memory); ends with a
 * block barrier */
__device__ inline void block_acc(payload_acc &a, unsigned long long nulls, unsigned long long (&sm)[5]) {
  if (threadIdx.x < 5) sm[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long mism = a.mism;   /* per lane 32 bits; summed over the warp in 64 */
  for (int o = 16; o; o >>= 1) {
    mism += __shfl_xor_sync(0xffffffffu, mism, o);
    a.x ^= __shfl_xor_sync(0xffffffffu, a.x, o);
    a.s += __shfl_xor_sync(0xffffffffu, a.s, o);
    a.words += __shfl_xor_sync(0xffffffffu, a.words, o);
    nulls += __shfl_xor_sync(0xffffffffu, nulls, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&sm[0], nulls);
    atomicAdd(&sm[1], mism);
    atomicXor(&sm[2], (unsigned long long)a.x);
    atomicAdd(&sm[3], a.s);
    atomicAdd(&sm[4], a.words);
  }
  __syncthreads();
}

/* A block's counters (block_acc) added to acc, the five words of an ouro_check
 * in their order.  The words checked are 32-bit, so their XOR only ever touches
 * the low half of its word; the high half may hold a fused round's task
 * counter. */
__device__ __forceinline__ void add_check(const unsigned long long (&sm)[5], unsigned long long *acc) {
  if (sm[0]) atomicAdd(&acc[0], sm[0]);
  if (sm[1]) atomicAdd(&acc[1], sm[1]);
  atomicXor(reinterpret_cast<unsigned *>(&acc[2]), (unsigned)sm[2]);
  atomicAdd(&acc[3], sm[3]);
  atomicAdd(&acc[4], sm[4]);
}

__device__ inline void flush_acc(payload_acc &a, unsigned long long nulls, ouro_check *out) {
  __shared__ unsigned long long sm[5];
  block_acc(a, nulls, sm);
  if (threadIdx.x == 0) add_check(sm, reinterpret_cast<unsigned long long *>(out));
}

/* A work slot (a 128-byte line): all zero between launches, and never used by
 * two launches at a time (who may use which: round_work in ouro_kernels.cu).
 * The blocks add their counters to acc; the last one to finish writes the
 * sums to *out and leaves the slot zero for the next launch, so a launch needs
 * no memset of its counters or its result.  A launch without a slot (null)
 * has *out zeroed before it begins, and adds to that. */
struct work_slot {
  unsigned next, pad;          /* tasks drawn; zero again after the last draw */
  unsigned long long acc[5];   /* nulls, mismatches, xor, sum, words */
  unsigned long long done;     /* blocks finished */
};
__device__ inline void finish_acc(payload_acc &a, unsigned long long nulls, work_slot *w, ouro_check *out) {
  __shared__ unsigned long long sm[5];
  block_acc(a, nulls, sm);
  if (threadIdx.x == 0) {
    add_check(sm, w ? w->acc : reinterpret_cast<unsigned long long *>(out));
    if (!w) return;
    __threadfence();
    if (atomicAdd(&w->done, 1ull) == gridDim.x - 1) {
      __threadfence();
      unsigned long long *o = reinterpret_cast<unsigned long long *>(out);   /* five words, in acc's order */
      unsigned long long r[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) r[k] = ld_rlx(&w->acc[k]);
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        o[k] = r[k];
        w->acc[k] = 0;
      }
      w->done = 0;
    }
  }
}


/* warp reduction of the check counters; lane 0 adds them to *out */
__device__ inline void warp_flush(payload_acc &a, unsigned long long nulls, ouro_check *out) {
  unsigned long long mism = a.mism;   /* per lane 32 bits; summed over the warp in 64 */
  for (int o = 16; o; o >>= 1) {
    mism += __shfl_xor_sync(0xffffffffu, mism, o);
    a.x ^= __shfl_xor_sync(0xffffffffu, a.x, o);
    a.s += __shfl_xor_sync(0xffffffffu, a.s, o);
    a.words += __shfl_xor_sync(0xffffffffu, a.words, o);
    nulls += __shfl_xor_sync(0xffffffffu, nulls, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (nulls) atomicAdd(&out->nulls, nulls);
    if (mism) atomicAdd(&out->mismatches, mism);
    atomicXor(&out->xor64, (unsigned long long)a.x);
    atomicAdd(&out->sum64, a.s);
    atomicAdd(&out->words, a.words);
  }
}

}  // namespace detail
}  // namespace ouro

#define OURO_DISPATCH(VAR, CALL)                                                 \
  switch (VAR) {                                                                 \
    case OURO_PAGE_ARRAY: { constexpr int V = OURO_PAGE_ARRAY; CALL; break; }   \
    case OURO_PAGE_VLIST: { constexpr int V = OURO_PAGE_VLIST; CALL; break; }   \
    case OURO_CHUNK_ARRAY: { constexpr int V = OURO_CHUNK_ARRAY; CALL; break; } \
    case OURO_CHUNK_VLIST: { constexpr int V = OURO_CHUNK_VLIST; CALL; break; } \
    case OURO_PAGE_VARRAY: { constexpr int V = OURO_PAGE_VARRAY; CALL; break; } \
    case OURO_CHUNK_VARRAY: { constexpr int V = OURO_CHUNK_VARRAY; CALL; break; } \
    default: return OURO_ENOTSUP;                                                \
  }

#endif
