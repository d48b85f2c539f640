"""Statistics of a lookup whose pages are in flight when its bags are gathered: a page found in
flight counts as a busy hit, so every distinct page of every bag is a hit or a busy hit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import Ctx  # noqa: E402

DEV = "cuda:0"


def test_pages_found_in_flight_are_counted():
    # one warp whose lookahead requests every page before the bag that holds it: 2 ms a
    # command, so the gather finds it in flight, or READY beside the bag's first pages
    dim, n_bags, pool = 1024, 8, 16                   # a row a page
    rows = n_bags * pool
    T = synth.table_normal(1, rows, dim)
    idx = np.argsort(synth.uniform01(2, rows)).astype(np.int64)
    off = synth.bags_fixed(n_bags, pool)
    out = torch.empty((n_bags, dim), dtype=torch.float32, device=DEV)
    d_idx, d_off = torch.from_numpy(idx).to(DEV), torch.from_numpy(off).to(DEV)
    with Ctx(T.nbytes, cache_bytes=4096 * 4096, ways=8, emu_latency_ns=2_000_000) as c:
        c.put(0, T)
        ag.agile_reset_stats(c.h)
        ag.agile_config_parallelism(c.h, 1)
        ag.agile_embedding_bag(c.h, 0, rows, dim, d_idx.data_ptr(), d_off.data_ptr(), n_bags, out.data_ptr(),
                               ag.AGILE_ASYNC, c.stream)
        torch.cuda.synchronize()
        c.check()
        st = c.stats()
        assert np.array_equal(out.cpu().numpy().view(np.uint32), oracle.embedding_bag(T, idx, off).view(np.uint32))
        assert st["misses"] == rows
        assert st["hits"] + st["busy_hits"] >= n_bags * pool, st
