"""Misses that find every way of their set in flight wait without taking the lines that others wait
for: BFS through a cache of 1/32 of the column array on a device of 80 us a command.

A claim that finds no victim is counted (eagain).  With two lines a warp a set of 8 ways has 4
reads in flight on average, all 8 in 5% of the claims (Poisson); the wait is at most about
270 us (480 reads in flight at 3.6 a us, and the latency), and a warp that waits makes
rounds of four claims, nine of them within the first 8 us and one per 8 us then: at most
0.05 x 4 x (9 + 33) = 8.4 claims a miss.  Warps that claim without pause take each other's
pages before their use, and both counts grow."""
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import numpy as np  # noqa: E402

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import PAGE, Ctx, round_page  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("mode", [ag.AGILE_SYNC, ag.AGILE_ASYNC])
def test_claims_without_a_victim(mode):
    n, off, cols = synth.rmat_csr(3, 18, 16)
    col0 = round_page(off.nbytes)
    lines = cols.nbytes // 32 // PAGE // 8 * 8
    level = torch.empty(n, dtype=torch.int32, device=DEV)
    edges = torch.zeros(1, dtype=torch.int64, device=DEV)
    with Ctx(col0 + cols.nbytes, cache_bytes=lines * PAGE, ways=8, wait_timeout_ns=60_000_000_000) as c:
        c.put(0, off)
        c.put(col0, cols)
        ag.agile_set_device_model(c.h, num_devices=4, emu_latency_ns=80_000, emu_device_read_gbps=3.7,
                                  emu_device_write_gbps=2.2)
        ag.agile_reset_stats(c.h)
        for src in synth.bfs_sources(3, off, 5):
            ag.agile_invalidate(c.h, c.stream)
            ag.agile_bfs(c.h, 0, col0, n, int(src), level.data_ptr(), edges.data_ptr(), mode, c.stream)
        torch.cuda.synchronize()
        c.check()
        want, scanned = oracle.bfs(off, cols, int(src))
        assert np.array_equal(level.cpu().numpy(), want) and int(edges.item()) == scanned
        st = c.stats()
        assert st["eagain"] <= 9 * st["misses"], (st["eagain"], st["misses"])
