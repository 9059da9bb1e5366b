"""A vertex table that a heap does not know, from before its reset or of another
heap: every free of it is a recorded bad free and the heap stays as it was."""
import numpy as np
import pytest

from gpu_helpers import assert_no_overlap, same_canonical_as_post_create, to_dev, torch_cuda
from paper_2504_18211_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CHUNK, BYTES = 1024, 64 << 20


@pytest.fixture(scope="module")
def P():
    import paper_2504_18211_gb300 as P
    from paper_2504_18211_gb300 import build
    build.build()
    P.load()
    return P


def lists_in(heap):
    """lists of every length: plain arrays of all classes, and segments"""
    from paper_2504_18211_gb300.graph import GraphRun
    torch = torch_cuda()
    nv = 400
    src = np.repeat(np.arange(nv, dtype=np.uint32), np.arange(nv) * 3 // 2)
    g = GraphRun(src, np.arange(src.size, dtype=np.uint32), nv)
    g.init(heap)
    g.insert(heap)
    torch.cuda.synchronize()
    assert g.ctl_dict() == {"appended": src.size, "failed": 0, "skipped": 0}
    return g


def untouched(P, st):
    return st["error_bits"] == P._binding.ERR_BAD_FREE and not sum(st["frees"]) and not sum(st["mallocs"]) and not sum(st["queued"])


@pytest.mark.parametrize("variant", ["page_array", "page_vlist", "chunk_array", "chunk_varray"])
def test_table_from_before_a_reset(P, variant):
    torch = torch_cuda()
    with P.Heap(BYTES, CHUNK, variant) as heap:
        g = lists_in(heap)
        heap.reset()
        g.free(heap)
        torch.cuda.synchronize()
        assert untouched(P, heap.stats())
        same_canonical_as_post_create(heap.snapshot(), BYTES // CHUNK)
        sizes = W.uniform_sizes(20000, 1, CHUNK, seed=W.SEED_BASE + 71)
        ptrs = heap.malloc(to_dev(sizes))
        torch.cuda.synchronize()
        p = ptrs.cpu().numpy().view(np.uint64)
        assert np.all(p != 0)
        assert_no_overlap(p, sizes, heap.base, BYTES, CHUNK)


@pytest.mark.parametrize("variant", ["page_array", "page_vlist", "chunk_array"])
def test_table_of_another_heap(P, variant):
    torch = torch_cuda()
    with P.Heap(BYTES, CHUNK, variant) as heap, P.Heap(BYTES, CHUNK, variant) as other:
        g = lists_in(heap)
        g.free(other)
        torch.cuda.synchronize()
        assert untouched(P, other.stats())
        same_canonical_as_post_create(other.snapshot(), BYTES // CHUNK)
        st = heap.stats()
        assert st["error_bits"] == 0 and sum(st["live"]) > 0   # its blocks are still allocated
