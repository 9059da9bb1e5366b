"""Fused rounds large enough for whole tasks of 32 requests: which blocks of a task
form a row and which go one at a time (lists of pages pace tasks of small blocks,
unstaged page arrays leave small shares out of the row) does not change a word."""
import numpy as np
import pytest

import oracle
from gpu_helpers import to_dev, torch_cuda
from paper_2504_18211_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 160007                 # more than 16 requests for each of the warps of a full grid


@pytest.fixture(scope="module")
def P():
    import paper_2504_18211_gb300 as P
    from paper_2504_18211_gb300 import build
    build.build()
    P.load()
    return P


def sizes_of(kind):
    r = W.rng(W.SEED_BASE + 81)
    if kind == "rests":                                     # no whole unit, words and tail bytes only
        return r.integers(0, 16, N).astype(np.uint32)
    if kind == "around":                                    # task totals on both sides of every limit (128 to 1100 units)
        lim = np.repeat(r.integers(4, 36, (N + 31) // 32), 32)[:N]
        return np.maximum(lim * 16 + r.integers(-17, 18, N), 0).astype(np.uint32)
    if kind == "one_large":                                 # one large block among 31 small ones
        s = r.integers(1, 200, N)
        s[::32] = r.integers(200, 8193, s[::32].size)
        return s.astype(np.uint32)
    if kind == "few_small":                                 # a few small blocks among large ones
        s = r.integers(1000, 2049, N)
        s[r.random(N) < 0.1] = r.integers(0, 257)
        return s.astype(np.uint32)
    s = r.integers(0, 300, N)                               # nulls: no class
    s[r.random(N) < 0.2] = 2 << 20
    return s.astype(np.uint32)


@pytest.mark.parametrize("variant,staging", [("page_array", False), ("page_array", True), ("page_vlist", False),
                                             ("page_vlist", True), ("page_varray", False), ("chunk_vlist", True)])
@pytest.mark.parametrize("kind", ["rests", "around", "one_large", "few_small", "nulls"])
def test_words(P, variant, staging, kind):
    from paper_2504_18211_gb300.batching import BatchRun
    torch = torch_cuda()
    sizes = sizes_of(kind)
    want = dict(oracle.expected_checksums(np.where(sizes > 1 << 20, 0, sizes), 0x91, 1), mismatches=0)
    want["nulls"] = int(((sizes == 0) | (sizes > 1 << 20)).sum())
    d = to_dev(sizes)
    with P.Heap(2 << 30, 8192, variant, staging=staging) as heap:
        for _ in range(3):                                  # a cold heap, then pages in use before
            assert P.check_to_dict(heap.round_fused(d, 0x91, 1)) == want
        run = BatchRun(sizes, np.array([0, N], np.uint64), seed=0x91)
        run.run(heap, "persistent")
        torch.cuda.synchronize()
        assert run.checks() == [want]
        st = heap.stats()
        assert st["error_bits"] == 0 and sum(st["live"]) == 0


@pytest.mark.parametrize("staging", [False, True])
def test_list_keeps_up_with_one_size(P, staging):
    """A list whose producers run ahead of its segments must not stay behind: rounds of one small size took 30 to 50
    times as long as on a virtualized array, and take about twice as long."""
    torch = torch_cuda()
    d = to_dev(W.single_size(1 << 20, 64))
    out = torch.zeros(5, dtype=torch.int64, device="cuda")
    us = {}
    for variant in ("page_varray", "page_vlist"):
        with P.Heap(1 << 30, 8192, variant, staging=staging) as heap:
            for _ in range(20):                             # until the heap holds a page for every request in flight
                heap.round_fused(d, 1, 1, out=out)
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(21)]
            ev[0].record()
            for e in ev[1:]:
                heap.round_fused(d, 1, 1, out=out)
                e.record()
            torch.cuda.synchronize()
            us[variant] = float(np.median([a.elapsed_time(b) * 1e3 for a, b in zip(ev, ev[1:])]))
    assert us["page_vlist"] < 10 * us["page_varray"], us
