"""What the serving loop leaves of sessions that are still growing when the steps
run out: the slot arrays name every one of them with its blocks and checksum,
in both forms and whether or not the grid holds all slots at once, so that a
program can take them over or free them."""
import numpy as np
import pytest

import oracle
from oracle.patterns import serving_schedule
from gpu_helpers import torch_cuda
from paper_2504_18211_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BLOCK, SEED = 4096, 0x5E59


@pytest.fixture(scope="module")
def P():
    import paper_2504_18211_gb300 as P
    from paper_2504_18211_gb300 import build
    build.build()
    P.load()
    return P


@pytest.mark.parametrize("form", ["persistent", "per_launch"])
@pytest.mark.parametrize("n_slots", [3, 700, 12000])        # 12000: more than a grid of 2 blocks per SM holds
@pytest.mark.parametrize("steps", [1, 7])
def test_unfinished_sessions(P, form, n_slots, steps):
    from paper_2504_18211_gb300.serving import ServeRun
    torch = torch_cuda()
    r = W.rng(W.SEED_BASE + 45)
    n = n_slots + n_slots // 3
    arrive = np.sort(r.integers(0, 4, n)).astype(np.uint32)
    blocks = r.integers(1, 12, n).astype(np.uint32)
    cap = 1 << 20
    admit, done, k = serving_schedule(arrive, blocks, steps, n_slots, cap)
    run = ServeRun(arrive, blocks, n_slots=n_slots, max_blocks=16, steps=steps, seed=SEED, block_bytes=BLOCK)
    for t in (run.slot_session, run.slot_k, run.slot_acc, run.tables):
        t.fill_(-7)
    with P.Heap(1 << 30, 16384, "page_array") as heap:
        run.run(heap, cap, form=form)
        sess = run.slot_session.cpu().numpy()
        slots = np.flatnonzero(sess >= 0)
        assert np.array_equal(np.sort(sess[slots]), np.flatnonzero((admit >= 0) & (done < 0)))
        assert np.all(sess[sess < 0] == -1)
        got_k = run.slot_k.cpu().numpy()[slots]
        assert np.array_equal(got_k, k[sess[slots]])
        acc = run.slot_acc.cpu().numpy().view(np.uint64).reshape(-1, 3)[slots]
        assert np.all(acc[:, 2] == 0)
        for i in range(0, slots.size, max(1, slots.size // 12)):
            want = oracle.expected_checksums(np.full(int(got_k[i]), BLOCK, np.uint32), SEED + int(sess[slots[i]]), 1)
            assert (int(acc[i, 0]), int(acc[i, 1])) == (want["xor64"], want["sum64"])
        tables = run.tables.view(n_slots, 16).cpu().numpy()
        live = np.concatenate([tables[s, :c] for s, c in zip(slots, got_k)] + [np.zeros(0, np.int64)])
        assert sum(heap.stats()["live"]) == live.size
        heap.free(torch.from_numpy(live).cuda())
        st = heap.stats()
        assert st["error_bits"] == 0 and sum(st["live"]) == 0
