"""The serving loop at the edges of its slot groups and payload pieces: blocks
of a few units, more slots than the grid holds at once, sessions of no blocks,
a single step, and a heap that is too small for what is admitted."""
import numpy as np
import pytest

import oracle
from oracle.patterns import serving_schedule
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


def run_both(P, arrive, blocks, n_slots, steps, block, heap_bytes, cap, variant="page_array"):
    from paper_2504_18211_gb300.serving import ServeRun
    torch_cuda()
    out = []
    for form in ("persistent", "per_launch"):
        run = ServeRun(arrive, blocks, n_slots=n_slots, max_blocks=64, steps=steps, seed=0x5E58, block_bytes=block)
        with P.Heap(heap_bytes, 16384, variant) as heap:
            run.run(heap, cap, form=form)
            r = run.results()
            st = heap.stats()
        assert r["error"] == 0 and st["error_bits"] == 0
        assert sum(st["live"]) == r["mallocs"] - r["frees"]
        out.append(r)
    return out


@pytest.mark.parametrize("block", [16, 48, 4096, 4112, 8208, 16384])
@pytest.mark.parametrize("n_slots,n", [(5, 40), (12000, 11000)])
def test_blocks_and_slots(P, block, n_slots, n):
    r = W.rng(W.SEED_BASE + 44)
    steps = 12
    arrive = np.sort(r.integers(0, 4, n)).astype(np.uint32)
    blocks = r.integers(1, 6, n).astype(np.uint32)
    cap = 1 << 20
    admit, done, k = serving_schedule(arrive, blocks, steps, n_slots, cap)
    for got in run_both(P, arrive, blocks, n_slots, steps, block, 1 << 30, cap):
        assert got["failed"] == 0
        assert np.array_equal(got["admit"], admit) and np.array_equal(got["done"], done)
        assert got["mallocs"] == int(k.sum()) and got["frees"] == int(blocks[done >= 0].sum())
        fin = np.flatnonzero(done >= 0)
        assert np.all(got["mism"][fin] == 0)
        for s in fin[:: max(1, fin.size // 12)]:
            want = oracle.expected_checksums(np.full(int(blocks[s]), block, np.uint32), 0x5E58 + int(s), 1)
            assert (int(got["xor"][s]), int(got["sum"][s])) == (want["xor64"], want["sum64"])


def test_empty_sessions_and_one_step(P):
    arrive = np.zeros(50, np.uint32)
    blocks = np.resize(np.array([0, 1, 3], np.uint32), 50)
    for steps in (1, 4):
        for got in run_both(P, arrive, blocks, 64, steps, 4096, 64 << 20, 1 << 20):
            done = np.where(blocks <= 1, 0, 2)
            assert np.all(got["admit"] == 0)
            assert np.array_equal(got["done"], np.where(done < steps, done, -1))
            assert got["frees"] == int(blocks[done < steps].sum())


def test_heap_smaller_than_what_is_admitted(P):
    """A growth that finds no memory counts as failed and is tried again in the next step."""
    arrive = np.zeros(100, np.uint32)
    blocks = np.resize(np.array([1, 2, 60], np.uint32), 100)
    for got in run_both(P, arrive, blocks, 128, 30, 16384, 1 << 20, 1 << 20):
        assert got["failed"] > 0 and got["mallocs"] - got["frees"] <= 64
        fin = got["done"] >= 0
        assert fin.sum() > 0 and np.all(got["mism"][fin] == 0)
