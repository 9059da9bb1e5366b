"""Appends to adjacency lists where the runs of a block meet their limits: one
source only, block edges, the step from the plain array to the segments, two
insertions at once on two streams, and a heap that runs out."""
import numpy as np
import pytest

from oracle.patterns import graph_class_counts
from gpu_helpers import torch_cuda
from paper_2504_18211_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2504_18211_gb300 as P
    from paper_2504_18211_gb300 import build
    build.build()
    P.load()
    return P


def check_rows(g, heap, src, dst, nv):
    deg, _, out = g.gather(heap)
    assert np.array_equal(deg, np.bincount(src, minlength=nv))
    got = np.lexsort((out, np.repeat(np.arange(nv), deg)))
    assert np.array_equal(out[got], dst[np.lexsort((dst, src))])
    return deg


@pytest.mark.parametrize("variant", ["page_array", "chunk_varray"])
@pytest.mark.parametrize("ne", [1, 31, 2047, 2048, 2049, 30000])
@pytest.mark.parametrize("nv", [1, 7, 4099])
def test_runs_at_their_limits(P, variant, ne, nv):
    from paper_2504_18211_gb300.graph import GraphRun
    torch = torch_cuda()
    r = W.rng(W.SEED_BASE + 53 + ne)
    src = r.integers(0, nv, ne).astype(np.uint32)
    dst = r.integers(0, 1 << 32, ne, dtype=np.uint64).astype(np.uint32)
    chunk = 256                                             # 64 entries, then segments of 62
    g = GraphRun(src, dst, nv)
    with P.Heap(64 << 20, chunk, variant) as heap:
        g.init(heap)
        g.insert(heap)
        torch.cuda.synchronize()
        assert g.ctl_dict() == {"appended": ne, "failed": 0, "skipped": 0}
        deg = check_rows(g, heap, src, dst, nv)
        st = heap.stats()
        m, f, _ = graph_class_counts(deg, chunk, heap.n_classes)
        assert st["mallocs"] == m.tolist() and st["frees"] == f.tolist() and st["error_bits"] == 0
        g.free(heap)
        torch.cuda.synchronize()
        assert sum(heap.stats()["live"]) == 0


@pytest.mark.parametrize("variant", ["page_array", "page_vlist"])
def test_two_insertions_at_once(P, variant):
    """Two halves of the edges on two streams, with the same hubs in both."""
    import ctypes as C
    from paper_2504_18211_gb300 import _binding as B
    from paper_2504_18211_gb300.graph import GraphRun
    torch = torch_cuda()
    nv, ne = 600, 1 << 17
    src, dst = W.graph_workload(n_vertices=nv, n_edges=ne, seed=W.SEED_BASE + 54)
    g = GraphRun(src, dst, nv)
    with P.Heap(256 << 20, 1024, variant) as heap:
        g.init(heap)
        torch.cuda.synchronize()
        for k in range(2):
            s = torch.cuda.Stream()
            h = slice(k * (ne // 2), (k + 1) * (ne // 2))
            B._check("ouro_graph_insert", B.load().ouro_graph_insert(
                C.c_void_p(heap.h), B._ptr(g.vt), B._ptr(g.d_src[h]), B._ptr(g.d_dst[h]), ne // 2, B._ptr(g.ctl),
                B._stream(s)))
        torch.cuda.synchronize()
        assert g.ctl_dict() == {"appended": ne, "failed": 0, "skipped": 0}
        check_rows(g, heap, src, dst, nv)
        assert heap.stats()["error_bits"] == 0


def test_full_heap_drops_what_does_not_fit(P):
    from paper_2504_18211_gb300.graph import GraphRun
    torch = torch_cuda()
    nv, ne = 64, 1 << 16
    r = W.rng(W.SEED_BASE + 55)
    src, dst = r.integers(0, nv, ne).astype(np.uint32), np.arange(ne, dtype=np.uint32)
    g = GraphRun(src, dst, nv)
    with P.Heap(128 << 10, 1024, "page_array") as heap:     # 128 KiB for 256 KiB of entries
        g.init(heap)
        g.insert(heap)
        torch.cuda.synchronize()
        c = g.ctl_dict()
        assert c["skipped"] == 0 and c["failed"] > 0 and c["appended"] + c["failed"] == ne
        deg, off, out = g.gather(heap)
        assert int(deg.sum()) == c["appended"]
        for v in range(nv):                                 # every kept entry is one of the vertex's edges, once
            row = out[off[v]:off[v + 1]]
            assert np.unique(row).size == row.size and np.all(src[row] == v)
        assert heap.stats()["error_bits"] == 0
