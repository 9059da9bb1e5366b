"""The calls whose speed this allocator is held to, and what one pass of each computes.

Every case is work that a program has the library do through its public entry
points.  Six kinds:

  fused     one ouro_round_fused launch: every request allocates, writes its
            pattern, reads it back and frees (a kernel that builds and drops
            its own temporaries);
  launches  the same round as the paper's driver runs it (Sec. 3 of arXiv
            2504.18211): ouro_batch_malloc, ouro_pattern_write,
            ouro_pattern_check and ouro_batch_free, one launch each (blocks
            that live from one kernel to the next);
  batches   many request batches of uneven size in one persistent kernel;
  replay    many small request batches as one CUDA graph of fused rounds;
  serve     sessions that grow block by block and finish, all steps of the
            request loop on the device;
  graph     adjacency lists that grow while edges arrive, are read back as
            rows and released.

Sizes of a request list: "single" (every request the same), "sweep" (2^k
bytes, k uniform), "uniform" (any byte count) and "mixed" (powers of two, odd
byte counts, runs above one chunk, empty and oversized requests).  A heap is
created once and then serves every pass, as in a program.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

import paper_2504_18211_gb300 as P
from paper_2504_18211_gb300 import _binding as B
from paper_2504_18211_gb300 import batching, graph, serving
from paper_2504_18211_gb300 import workloads as W

MIB = 1 << 20
CHUNK = 8192
GOLD = 0x9E3779B9
BLOCK = 16384            # bytes of a serving block


def listed():
    return [
        # the paper's small plain run: 40 x 256 threads, 16 bytes each, in one launch
        {"name": "small_fused", "kind": "fused", "variant": "page_array", "staging": False, "n": 10240,
         "sizes": "single", "lo": 16, "hi": 16, "mode": 1, "heap_mib": 64},
        # the paper's axis of 1024 threads of 1000 bytes, one launch per phase: launch latency counts
        {"name": "small_launches", "kind": "launches", "variant": "page_array", "n": 1024,
         "sizes": "single", "lo": 1000, "hi": 1000, "mode": 1, "heap_mib": 64},
        # the size sweep that the benchmark reports: temporaries of every size class in one kernel
        {"name": "sweep_fused", "kind": "fused", "variant": "page_array", "staging": True, "n": 1 << 20,
         "sizes": "sweep", "lo": 16, "hi": 8192, "mode": 1, "heap_mib": 8192},
        # the same sweep as the paper's driver: blocks that outlive the kernel that allocated them
        {"name": "sweep_launches", "kind": "launches", "variant": "page_array", "n": 1 << 20,
         "sizes": "sweep", "lo": 16, "hi": 8192, "mode": 1, "heap_mib": 8192},
        # allocation itself: every kind of request, one word stored in each block (the paper's thread id)
        {"name": "mixed_ids_launches", "kind": "launches", "variant": "page_array", "n": (1 << 20) - 77,
         "sizes": "mixed", "lo": 0, "hi": 65536, "mode": 0, "heap_mib": 8192},
        # chunk queues, the form that wastes no memory on fixed pages, at a ragged size
        {"name": "mixed_ids_chunk", "kind": "launches", "variant": "chunk_array", "n": 300007,
         "sizes": "mixed", "lo": 0, "hi": 65536, "mode": 0, "heap_mib": 4096},
        # chunk queues inside a kernel that also frees
        {"name": "sweep_fused_chunk", "kind": "fused", "variant": "chunk_varray", "staging": True, "n": 200003,
         "sizes": "sweep", "lo": 16, "hi": 8192, "mode": 1, "heap_mib": 2048},
        # a burst of one size on queues that keep their storage inside the heap
        {"name": "burst_vlist", "kind": "launches", "variant": "page_vlist", "n": 3 << 18,
         "sizes": "single", "lo": 64, "hi": 64, "mode": 1, "heap_mib": 2048},
        # a stream of uneven batches, every batch's temporaries of any byte count
        {"name": "batches_persistent", "kind": "batches", "variant": "page_array", "staging": True, "n_batches": 96,
         "log_lo": 10, "log_hi": 18, "hi": 8192, "heap_mib": 8192},
        # small batches at interactive rates: one replayed graph
        {"name": "batches_replay", "kind": "replay", "variant": "page_array", "staging": False, "n_batches": 32,
         "log_lo": 8, "log_hi": 13, "hi": 4096, "heap_mib": 1024},
        # a serving loop at a load that now and then fills its slots, from the first arrival to the last free
        {"name": "serving_loop", "kind": "serve", "variant": "page_array", "steps": 400, "rate": 5500,
         "median_kib": 1024, "slots": 4096, "heap_mib": 16384},
        # a scale-free graph arriving edge by edge
        {"name": "graph_growth", "kind": "graph", "variant": "page_array", "vertices": 1 << 18, "edges": 1 << 22,
         "heap_mib": 2048},
    ]


def _log(rng, lo, hi):
    """A whole number whose logarithm is uniform over [lo, hi]."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(("fused", "fused", "launches", "launches", "launches", "batches", "replay", "serve", "graph"))
    variant = rng.choice(("page_array", "page_array", "page_vlist", "page_varray", "chunk_array", "chunk_varray",
                          "chunk_vlist"))
    staging = rng.random() < 0.5
    if kind in ("fused", "launches"):
        n = _log(rng, 1000, 1 << 20)
        sizes = rng.choice(("single", "sweep", "uniform", "mixed"))
        lo, hi = {"single": (16, 2048), "sweep": (16, 8192), "uniform": (1, 8192), "mixed": (0, 65536)}[sizes]
        if sizes == "single":
            lo = hi = _log(rng, lo, hi)
        # room for every request at its class, twice over, for the queues' own chunks and for runs
        heap = 64 + 2 * n * {"single": 2 * hi, "sweep": 2048, "uniform": 8192, "mixed": 6144}[sizes] // MIB
        case = {"kind": kind, "variant": variant, "n": n, "sizes": sizes, "lo": lo, "hi": hi,
                "mode": 0 if sizes == "mixed" and rng.random() < 0.5 else 1, "heap_mib": heap}
        if kind == "fused":
            case["staging"] = staging
        return case
    if kind == "batches":
        return {"kind": kind, "variant": variant, "staging": staging, "n_batches": _log(rng, 8, 64), "log_lo": 8,
                "log_hi": rng.randint(12, 17), "hi": _log(rng, 64, 8192), "heap_mib": 4096}
    if kind == "replay":
        return {"kind": kind, "variant": variant, "staging": staging, "n_batches": _log(rng, 8, 64), "log_lo": 6,
                "log_hi": rng.randint(10, 13), "hi": _log(rng, 64, 8192), "heap_mib": 1024}
    if kind == "serve":
        case = {"kind": kind, "variant": rng.choice(("page_array", "page_array", "page_varray", "chunk_array")),
                "steps": _log(rng, 50, 400), "median_kib": _log(rng, 64, 1024), "slots": _log(rng, 256, 4096),
                "heap_mib": 16384}
        case["rate"] = round(100 * case["slots"] / _mean_blocks(case) * rng.uniform(0.2, 0.95))   # of what the slots take
        return case
    return {"kind": "graph", "variant": rng.choice(("page_array", "page_array", "page_varray", "chunk_array")),
            "vertices": _log(rng, 1 << 14, 1 << 18), "edges": _log(rng, 1 << 16, 1 << 21), "heap_mib": 2048}


# ------------------------------------------------------------------ inputs
def _sizes(case, seed):
    n, lo, hi = case["n"], case["lo"], case["hi"]
    if case["sizes"] == "single":
        return W.single_size(n, hi)
    if case["sizes"] == "sweep":
        return W.sweep_sizes(n, seed=seed, kmin=lo.bit_length() - 1, kmax=hi.bit_length() - 1)
    if case["sizes"] == "uniform":
        return W.uniform_sizes(n, lo, hi, seed=seed)
    return W.mixed_sizes(n, seed=seed, chunk_bytes=CHUNK)


def _batches(case, seed):
    return W.batching_workload(n_batches=case["n_batches"], lo=case["log_lo"], hi=case["log_hi"], smin=4,
                               smax=case["hi"], seed=seed)


def _sessions(case, seed):
    """Sessions of workloads.serving_workload's kind that a run of `steps` steps serves to their end: a given number
    of them, arriving in the first 40 % of the steps and growing for at most 40 % of them."""
    r = W.rng(seed)
    span = case["steps"] * 2 // 5
    n = int(case["rate"] * 0.01 * span)
    arrive = np.sort(r.integers(0, span, n)).astype(np.uint32)
    size = r.lognormal(math.log(case["median_kib"] << 10), 1.0, n)
    return arrive, np.clip(np.ceil(size / BLOCK), 1, span).astype(np.uint32)


def _mean_blocks(case):
    """Mean of ceil(lognormal / BLOCK) clipped to the 40 % of the steps, by quadrature over the quantiles."""
    q = [(i + 0.5) / 400 for i in range(400)]
    z = [math.sqrt(2.0) * _erfinv(2 * p - 1) for p in q]
    span = case["steps"] * 2 // 5
    return sum(min(max(math.ceil((case["median_kib"] << 10) * math.exp(t) / BLOCK), 1), span) for t in z) / len(z)


def _erfinv(x):
    """Winitzki's approximation (2 parts in 1000), enough for an expected size."""
    a, ln = 0.147, math.log(1 - x * x)
    t = 2 / (math.pi * a) + ln / 2
    return math.copysign(math.sqrt(math.sqrt(t * t - ln / a) - t), x)


def _edges(case, seed):
    return W.graph_workload(case["vertices"], case["edges"], seed=seed)


def _pattern_seed(seed):
    return (seed * 2654435761 + 12345) & 0x7FFFFFFF


def prepare(case, seed):
    kind, variant = case["kind"], case["variant"]
    chunk = BLOCK if kind == "serve" else CHUNK
    st = {"case": case, "seed": _pattern_seed(seed),
          "heap": P.Heap(case["heap_mib"] * MIB, chunk, variant, staging=bool(case.get("staging", False)))}
    if kind in ("fused", "launches"):
        st["sizes"] = torch.from_numpy(_sizes(case, seed).view(np.int32)).cuda()
        st["ptrs"] = torch.empty(case["n"], dtype=torch.int64, device="cuda")
        st["out"] = torch.zeros(5, dtype=torch.int64, device="cuda")
    elif kind in ("batches", "replay"):
        sizes, offs = _batches(case, seed)
        st["run"] = batching.BatchRun(sizes, offs, seed=st["seed"])
    elif kind == "serve":
        arrive, blocks = _sessions(case, seed)
        st["cap"] = int(0.95 * (case["heap_mib"] * MIB // BLOCK))
        st["run"] = serving.ServeRun(arrive, blocks, n_slots=case["slots"], max_blocks=int(blocks.max(initial=1)),
                                     steps=case["steps"], seed=st["seed"], block_bytes=BLOCK)
    else:
        src, dst = _edges(case, seed)
        st["run"] = graph.GraphRun(src, dst, case["vertices"])
        st["vertex"] = torch.arange(case["vertices"], device="cuda")
        st["rows"] = torch.empty(case["edges"], dtype=torch.int32, device="cuda")
    return st


# --------------------------------------------------------------- one pass
def run(state):
    kind, heap = state["case"]["kind"], state["heap"]
    if kind == "fused":
        return heap.round_fused(state["sizes"], state["seed"], state["case"]["mode"], out=state["out"])
    if kind == "launches":
        sizes, ptrs, mode = state["sizes"], state["ptrs"], state["case"]["mode"]
        heap.malloc(sizes, ptrs)
        P.pattern_write(ptrs, sizes, state["seed"], mode)
        P.pattern_check(ptrs, sizes, state["seed"], mode, out=state["out"])
        heap.free(ptrs)
        return state["out"]
    r = state["run"]
    if kind == "batches":
        r.run(heap, "persistent")
        return r.out
    if kind == "replay":
        r.run(heap, "graph")
        return r.out
    if kind == "serve":
        r.run(heap, state["cap"])
        return {"sessions": r.sess_out.view(-1, 5), "counts": r.ctl[5:8]}   # counts: mallocs, frees, failed
    # the entries of a row stand in the order in which the edges won their
    # vertex, so the program sorts each row before it keeps it
    r.init(heap)
    r.insert(heap)
    degrees = r.vt.view(torch.int32).view(r.nv, r.vbytes // 4)[:, 8]
    offsets = torch.cumsum(degrees, 0, dtype=torch.int64) - degrees
    B._check("ouro_graph_gather", B.load().ouro_graph_gather(
        C.c_void_p(heap.h), B._ptr(r.vt), r.nv, B._ptr(offsets), B._ptr(state["rows"]), B._stream(None)))
    r.free(heap)
    owner = torch.repeat_interleave(state["vertex"], degrees, output_size=r.ne)
    rows = torch.sort((owner << 32) | state["rows"])[0]
    return {"degrees": degrees, "rows": rows, "counts": r.ctl}


# ------------------------------------------------------------------- work
def _mean_size(case):
    """Expected bytes of payload per request."""
    lo, hi, kind = case["lo"], case["hi"], case["sizes"]
    if kind == "single":
        return float(hi)
    if kind == "uniform":
        return (lo + hi) / 2
    ks = range(4, 14) if kind == "mixed" else range(lo.bit_length() - 1, hi.bit_length())
    sweep = sum(2.0 ** k for k in ks) / len(ks)
    return sweep if kind == "sweep" else 0.64 * sweep + 0.30 * CHUNK / 2 + 0.02 * (CHUNK + 65536) / 2


def work(case):
    kind = case["kind"]
    if kind in ("fused", "launches"):
        n = case["n"]
        per = 4 if kind == "fused" else 24     # the size; the pointers written once and read three times
        pay = _mean_size(case) if case["mode"] else 4.0
        return {"bytes": n * (per + pay * (1 if kind == "fused" else 2)), "flops": 0}
    if kind in ("batches", "replay"):
        lo, hi = case["log_lo"], case["log_hi"]
        mean = (2.0 ** hi - 2.0 ** lo) / ((hi - lo) * math.log(2))
        return {"bytes": case["n_batches"] * (40 + mean * (4 + (4 + case["hi"]) / 2)), "flops": 0}
    if kind == "serve":
        n = int(case["rate"] * 0.01 * (case["steps"] * 2 // 5))
        return {"bytes": n * (48 + _mean_blocks(case) * (BLOCK + 8)), "flops": 0}
    # the edges read, the rows written, read and written again in order, the vertex records
    return {"bytes": case["edges"] * (8 + 4 + 8 + 8) + case["vertices"] * 40, "flops": 0}


# ------------------------------------------------------------------ exact
def _fmix32(x):
    x = x.astype(np.uint32)
    x ^= x >> np.uint32(16)
    x *= np.uint32(0x85EBCA6B)
    x ^= x >> np.uint32(13)
    x *= np.uint32(0xC2B2AE35)
    x ^= x >> np.uint32(16)
    return x


def _check_of(sizes, seed, mode):
    """nulls, mismatches, xor, sum and count of the words that a round reads back."""
    ids = np.arange(sizes.size, dtype=np.uint32)
    live = (sizes > 0) & (sizes <= MIB)
    nulls = int(sizes.size - live.sum())
    if mode == 0:
        t = ids[live]
        return [nulls, 0, int(np.bitwise_xor.reduce(t)) if t.size else 0, int(t.sum(dtype=np.uint64)), int(t.size)]
    keys = _fmix32(np.uint32(seed & 0xFFFFFFFF) ^ (ids * np.uint32(GOLD)))[live]
    size = sizes[live]
    order = np.argsort(size, kind="stable")
    keys, full, tail = keys[order], (size[order] >> 2).astype(np.int64), (size[order] & 3).astype(np.uint32)
    part = tail > 0
    last = (keys[part] + full[part].astype(np.uint32) * np.uint32(GOLD)) & ((np.uint32(1) << (8 * tail[part])) - np.uint32(1))
    xor = int(np.bitwise_xor.reduce(last)) if last.size else 0
    total = int(last.sum(dtype=np.uint64))
    at = 0
    while at < keys.size:
        end = min(keys.size, at + max(1, (4 << 20) // max(1, int(full[at]))))
        while end > at + 1 and (end - at) * int(full[end - 1]) > (8 << 20):
            end = at + (end - at) // 2
        w = np.arange(int(full[end - 1]), dtype=np.uint32) * np.uint32(GOLD)
        v = keys[at:end, None] + w[None, :]
        v[np.arange(w.size)[None, :] >= full[at:end, None]] = 0
        if v.size:
            xor ^= int(np.bitwise_xor.reduce(v, axis=None))
            total += int(v.sum(dtype=np.uint64))
        at = end
    return [nulls, 0, xor, total, int(full.sum() + part.sum())]


def exact(case, seed):
    kind, key = case["kind"], _pattern_seed(seed)
    if kind in ("fused", "launches"):
        sizes = _sizes(case, seed)
        if case["mode"] and int(sizes.astype(np.int64).sum()) > (2 << 30):
            return None
        return np.array(_check_of(sizes, key, case["mode"]), dtype=np.int64)
    if kind in ("batches", "replay"):
        sizes, offs = _batches(case, seed)
        if int(sizes.astype(np.int64).sum()) > (2 << 30):
            return None
        offs = offs.astype(np.int64)
        return np.array([_check_of(sizes[offs[b]:offs[b + 1]], key + b, 1) for b in range(case["n_batches"])],
                        dtype=np.int64)
    if kind == "graph":
        src, dst = _edges(case, seed)
        rows = np.sort((src.astype(np.int64) << 32) | dst)
        return {"degrees": np.bincount(src, minlength=case["vertices"]).astype(np.int32), "rows": rows,
                "counts": np.array([case["edges"], 0, 0, 0], dtype=np.int64)}
    return None
