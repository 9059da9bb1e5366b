"""Fused rounds in flight together: a long round beside many short ones, replayed
graphs beside live rounds, and more streams than a heap has work slots.  Every
result is its own round's, and so is every result of the lone rounds after."""
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


SHORT = [1, 9, 300, 4000, 20011]           # grids of 1 block up to all of them
SEED = 0x510


@pytest.fixture(scope="module")
def short():
    """(device sizes, expected check) of a few short rounds; round k uses seed SEED + k"""
    out = []
    for k, n in enumerate(SHORT):
        s = W.uniform_sizes(n, 1, 600, seed=W.SEED_BASE + 61 + k)
        out.append((to_dev(s), dict(oracle.expected_checksums(s, SEED + k, 1), nulls=0, mismatches=0)))
    return out


class Rounds:
    """Rounds issued now, their results looked at later."""

    def __init__(self, P, heap, short):
        self.P, self.heap, self.short, self.todo = P, heap, short, []

    def issue(self, k, stream=None):
        torch = torch_cuda()
        out = torch.full((5,), -1, dtype=torch.int64, device="cuda")
        if stream is not None:
            stream.wait_stream(torch.cuda.current_stream())   # the fill above
        self.heap.round_fused(self.short[k][0], SEED + k, 1, out=out, stream=stream)
        self.todo.append((k, out))
        return out

    def check(self):
        torch_cuda().cuda.synchronize()
        for i, (k, out) in enumerate(self.todo):
            assert self.P.check_to_dict(out) == self.short[k][1], i
        self.todo = []

    def lone(self):
        """more rounds than work slots, one at a time"""
        for i in range(70):
            self.issue(i % len(SHORT))
            torch_cuda().cuda.synchronize()
        self.check()


@pytest.mark.parametrize("variant,staging", [("page_array", False), ("page_vlist", True), ("chunk_array", False)])
def test_long_round_beside_short_ones(P, short, variant, staging):
    torch = torch_cuda()
    n = 1 << 22
    sizes = np.full(n, 16, np.uint32)
    want = dict(oracle.expected_checksums(sizes, 5, 1), nulls=0, mismatches=0)
    d = to_dev(sizes)
    with P.Heap(1 << 30, 8192, variant, staging=staging) as heap:
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        r = Rounds(P, heap, short)
        longs = [torch.full((5,), -1, dtype=torch.int64, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        for out in longs:
            heap.round_fused(d, 5, 1, out=out, stream=a)
            for i in range(70):
                r.issue(i % len(SHORT), b)
        r.check()
        for out in longs:
            assert P.check_to_dict(out) == want
        r.lone()
        st = heap.stats()
        assert st["error_bits"] == 0 and sum(st["live"]) == 0


def test_graphs_beside_live_rounds(P, short):
    from paper_2504_18211_gb300.batching import BatchRun
    torch = torch_cuda()
    sizes, offs = W.batching_workload(n_batches=80, lo=0, hi=12, smax=700, seed=W.SEED_BASE + 62)
    runs = [BatchRun(sizes, offs, seed=900 + 100 * k) for k in range(2)]
    want = [[dict(oracle.expected_checksums(sizes[int(offs[b]):int(offs[b + 1])], run.seed + b, 1), nulls=0,
                  mismatches=0) for b in range(run.nb)] for run in runs]
    with P.Heap(1 << 30, 8192, "page_array") as heap:
        streams = [torch.cuda.Stream() for _ in range(4)]
        r = Rounds(P, heap, short)
        outs = [torch.full((5,), -1, dtype=torch.int64, device="cuda") for _ in SHORT]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[0]):           # a program's own capture
            for k, out in enumerate(outs):
                heap.round_fused(short[k][0], SEED + k, 1, out=out)
        torch.cuda.synchronize()
        for rep in range(4):
            with torch.cuda.stream(streams[0]):
                g.replay()
            for k, run in enumerate(runs):
                with torch.cuda.stream(streams[1 + k]):
                    run.run(heap, "graph")
            for i in range(40):
                r.issue(i % len(SHORT), streams[3])
        r.check()
        for k, out in enumerate(outs):
            assert P.check_to_dict(out) == short[k][1]
        for run, w in zip(runs, want):
            assert run.checks() == w
        r.lone()
        for run in runs:
            run.close()
        assert heap.stats()["error_bits"] == 0


def test_more_streams_than_slots(P, short):
    torch = torch_cuda()
    with P.Heap(1 << 30, 8192, "page_array") as heap:
        r = Rounds(P, heap, short)
        streams = [torch.cuda.ExternalStream(torch.cuda.Stream(priority=-(i & 1)).cuda_stream) for i in range(64)]
        import ctypes as C
        rt = C.CDLL("libcudart.so.13")
        own = []
        for _ in range(80):                                    # PyTorch hands its streams out again: streams of our own
            h = C.c_void_p()
            assert rt.cudaStreamCreateWithFlags(C.byref(h), 1) == 0
            own.append(h)
        streams += [torch.cuda.ExternalStream(h.value) for h in own]
        for rep in range(2):
            for i, s in enumerate(streams):
                r.issue((i + rep) % len(SHORT), s)
        r.check()
        r.lone()
        for h in own:
            assert rt.cudaStreamDestroy(h) == 0
        st = heap.stats()
        assert st["error_bits"] == 0 and sum(st["live"]) == 0
