"""Payload rows: blocks of every length around the edges of a row unit, of the
row itself and of a task, written and read back fused and per launch, against
the oracle's checksums (whole numbers: equality)."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2504_18211_gb300 as P  # noqa: E402

EDGES = [1, 3, 4, 15, 16, 17, 31, 32, 33, 255, 256, 257, 271, 272, 273, 1008, 1024, 1025, 1039, 1040, 1041, 2048, 8191,
         8192]


def sizes_of(kind: str, n: int) -> np.ndarray:
    if kind == "edges":
        return np.resize(np.array(EDGES, np.uint32), n)
    if kind == "sorted":
        return np.sort(np.resize(np.array(EDGES, np.uint32), n))
    return np.full(n, {"units": 16, "rest": 7, "row": 256}[kind], np.uint32)


@pytest.mark.parametrize("kind", ["edges", "sorted", "units", "rest", "row"])
@pytest.mark.parametrize("n", [1, 31, 33, 4097, 70001])
def test_rows(kind, n):
    sizes = sizes_of(kind, n)
    d = torch.from_numpy(sizes.view(np.int32)).cuda()
    for mode in (1, 0):
        want = dict(oracle.expected_checksums(sizes, 0x77, mode), nulls=0, mismatches=0)
        with P.Heap(1 << 30, 8192, "page_array", staging=bool(n & 2)) as heap:
            p = heap.malloc(d)
            P.pattern_write(p, d, 0x77, mode)
            assert P.check_to_dict(P.pattern_check(p, d, 0x77, mode)) == want
            P.pattern_write(p, d, 0x78, 1)                  # other words: every one of them is seen
            got = P.check_to_dict(P.pattern_check(p, d, 0x77, 1))
            assert got["nulls"] == 0 and got["mismatches"] > 0 and got["words"] == int(((sizes + 3) // 4).sum())
            heap.free(p)
            assert P.check_to_dict(heap.round_fused(d, 0x77, mode)) == want
            assert heap.stats()["error_bits"] == 0


def test_work_slots_come_back_empty():
    """More rounds than work slots, of changing size, on two streams: every result is its own round's."""
    with P.Heap(256 << 20, 8192, "page_array") as heap:
        streams = [torch.cuda.Stream() for _ in range(2)]
        runs = []
        for k in range(140):
            sizes = sizes_of("edges", 1 + 37 * k)
            d = torch.from_numpy(sizes.view(np.int32)).cuda()
            out = torch.full((5,), -1, dtype=torch.int64, device="cuda")
            runs.append((sizes, d, out))
        torch.cuda.synchronize()
        for k, (_, d, out) in enumerate(runs):
            heap.round_fused(d, k, 1, out=out, stream=streams[k & 1])
        empty = heap.round_fused(runs[0][1][:0], 1, 1)
        torch.cuda.synchronize()
        for k, (sizes, _, out) in enumerate(runs):
            assert P.check_to_dict(out) == dict(oracle.expected_checksums(sizes, k, 1), nulls=0, mismatches=0)
        assert P.check_to_dict(empty) == dict(nulls=0, mismatches=0, xor64=0, sum64=0, words=0)
        heap.reset()
        sizes, d, out = runs[3]
        assert P.check_to_dict(heap.round_fused(d, 3, 1, out=out))["xor64"] == \
            oracle.expected_checksums(sizes, 3, 1)["xor64"]
