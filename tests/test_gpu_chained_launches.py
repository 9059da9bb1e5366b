"""Kernels that are set up while their predecessor runs: behind copies, fills
and other kernels, on one stream and after an event of another, eagerly and in
a captured graph, every result is that of the calls in order."""
import numpy as np
import pytest

import oracle
from gpu_helpers import to_dev, torch_cuda
from paper_2504_18211_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2504_18211_gb300 as P
    from paper_2504_18211_gb300 import build
    build.build()
    P.load()
    return P


@pytest.mark.parametrize("variant", ["page_array", "chunk_array", "page_vlist"])
@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("n", [700, 40001])
def test_calls_in_order(P, variant, captured, n):
    torch = torch_cuda()
    a, b = (W.uniform_sizes(n, 1, 4096, seed=W.SEED_BASE + 91 + k) for k in range(2))
    da, db = to_dev(a), to_dev(b)
    want = [dict(oracle.expected_checksums(s, 7, 1), nulls=0, mismatches=0) for s in (a, b)]
    sizes = torch.zeros(n, dtype=torch.int32, device="cuda")
    ptrs = torch.zeros(n, dtype=torch.int64, device="cuda")
    outs = [torch.zeros(5, dtype=torch.int64, device="cuda") for _ in range(4)]
    keep = torch.zeros(n, dtype=torch.int64, device="cuda")
    with P.Heap(1 << 30, 8192, variant) as heap:
        main, side = torch.cuda.Stream(), torch.cuda.Stream()

        def calls():
            sizes.copy_(da)                                 # a copy, then a chained kernel that reads it
            heap.round_fused(sizes, 7, 1, out=outs[0])
            heap.malloc(sizes, ptrs)
            P.pattern_write(ptrs, sizes, 7, 1)
            P.pattern_check(ptrs, sizes, 7, 1, out=outs[1])
            keep.copy_(ptrs)
            heap.free(ptrs)
            ptrs.zero_()                                    # after the free has read them
            sizes.copy_(db)                                 # after the check has read them
            heap.round_fused(sizes, 7, 1, out=outs[2])
            ev = torch.cuda.Event()
            ev.record(main)
            side.wait_event(ev)
            with torch.cuda.stream(side):
                heap.round_fused(sizes, 7, 1, out=outs[3])
            ev2 = torch.cuda.Event()
            ev2.record(side)
            main.wait_event(ev2)
            sizes.zero_()

        with torch.cuda.stream(main):
            calls()
        torch.cuda.synchronize()
        if captured:
            for o in outs:
                o.fill_(-1)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=main):
                calls()
            for _ in range(3):
                g.replay()
            torch.cuda.synchronize()
        for k, o in enumerate(outs):
            assert P.check_to_dict(o) == want[k >= 2], k
        assert bool((keep != 0).all()) and not bool(ptrs.any())
        st = heap.stats()
        assert st["error_bits"] == 0 and sum(st["live"]) == 0
