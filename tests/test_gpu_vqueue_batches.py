"""Large batches on virtualized page queues: the shares of a block cut across
segments of every length, several classes and runs at once, null pointers
among the frees, checked heaps, and a heap that runs out."""
import numpy as np
import pytest

from gpu_helpers import assert_no_overlap, per_class_counts, same_canonical_as_post_create, to_dev, torch_cuda
from paper_2504_18211_gb300 import workloads as W

pytestmark = pytest.mark.gpu
WIDE = 4 * 256 * 152            # requests from which a batch gives each thread four


@pytest.fixture(scope="module")
def ouro():
    import paper_2504_18211_gb300 as P
    from paper_2504_18211_gb300 import build
    build.build()
    P.load()
    return P


def sizes_of(kind, n):
    if kind == "single":
        return W.single_size(n, 16)
    return W.mixed_sizes(n, seed=W.SEED_BASE + 81) if kind == "mixed" else W.sweep_sizes(n, W.SEED_BASE + 82, 4, 8)


@pytest.mark.parametrize("variant", ["page_vlist", "page_varray"])
@pytest.mark.parametrize("kind,chunk,checked", [("single", 256, False), ("single", 8192, False), ("small", 512, False),
                                                ("mixed", 8192, False), ("mixed", 4096, True)])
@pytest.mark.parametrize("extra", [0, 1023])
def test_batches_across_segments(ouro, variant, kind, chunk, checked, extra):
    torch_cuda()
    n, seed = WIDE + extra, 0x51
    sizes = sizes_of(kind, n)
    live = (sizes > 0) & (sizes <= 1 << 20)
    heap_bytes = (2 << 30) if kind == "mixed" else (128 << 20)
    d = to_dev(sizes)
    with ouro.Heap(heap_bytes, chunk, variant, checked=checked) as heap:
        for _ in range(3):                              # the second and third on recycled segments
            ptrs = heap.malloc(d)
            ouro.pattern_write(ptrs, d, seed, 1)
            got = ouro.check_to_dict(ouro.pattern_check(ptrs, d, seed, 1))
            assert got["mismatches"] == 0 and got["nulls"] == int((~live).sum())
            assert got["words"] == int(((sizes[live].astype(np.int64) + 3) // 4).sum())
            p = ptrs.cpu().numpy().view(np.uint64)
            assert np.array_equal(p != 0, live)
            assert_no_overlap(p, sizes, heap.base, heap_bytes, chunk)
            heap.free(ptrs)                             # nulls among them
        st = heap.stats()
        assert st["error_bits"] == 0 and sum(st["live"]) == 0
        assert st["mallocs"] == [3 * c for c in per_class_counts(sizes, chunk)] == st["frees"]
        heap.trim()
        same_canonical_as_post_create(heap.snapshot(), heap_bytes // chunk)


@pytest.mark.parametrize("variant", ["page_vlist", "page_varray"])
def test_batch_larger_than_the_heap(ouro, variant):
    torch = torch_cuda()
    n = WIDE + 5
    d = to_dev(W.single_size(n, 1024))
    with ouro.Heap(64 << 20, 8192, variant, spin_limit=4000, backoff_max_ns=256) as heap:
        ptrs = heap.malloc(d)
        torch.cuda.synchronize()
        p = ptrs.cpu().numpy().view(np.uint64)
        ok = int((p != 0).sum())
        assert 0 < ok <= (64 << 20) // 1024 and np.unique(p[p != 0]).size == ok
        st = heap.stats()
        assert sum(st["mallocs"]) == ok and sum(st["failed"]) == n - ok
        heap.free(ptrs)
        torch.cuda.synchronize()
        assert sum(heap.stats()["live"]) == 0
