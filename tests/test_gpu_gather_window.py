"""The pages that all warps of a lookup request ahead of their use fit the queues: a cold pipeline
call and a cold embedding bag at the full grid, every row a miss, find a queue slot for each."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import Ctx, dyadic_rows, fill_dyadic  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("call", ["pipeline", "bag"])
def test_queues_hold_the_windows(call):
    # 2,048 warps with the cache's 32 rows each would request 65,536 pages on 4,032 slots
    rows, dim, n_bags, pool = 1 << 20, 64, 2048, 64
    idx = synth.indices_uniform(1, n_bags * pool, rows)
    d_idx = torch.from_numpy(idx).to(DEV)
    d_off = torch.from_numpy(synth.bags_fixed(n_bags, pool)).to(DEV)
    out = torch.empty((n_bags, dim), dtype=torch.float32, device=DEV)
    with Ctx(rows * dim * 4, cache_bytes=640 << 20, ways=8, num_queues=64, queue_depth=64) as c:
        fill_dyadic(c, 1, rows, dim, rows * dim * 4)
        ag.agile_reset_stats(c.h)
        if call == "pipeline":
            ag.agile_embedding_pipeline(c.h, 0, rows * dim * 4, 1, rows, dim, d_idx.data_ptr(), pool, n_bags, 1, 0,
                                        out.data_ptr(), ag.AGILE_SYNC, c.stream)
        else:
            ag.agile_embedding_bag(c.h, 0, rows, dim, d_idx.data_ptr(), d_off.data_ptr(), n_bags, out.data_ptr(),
                                   ag.AGILE_SYNC, c.stream)
        torch.cuda.synchronize()
        c.check()
        st = c.stats()
        want = dyadic_rows(0, idx, dim).reshape(n_bags, pool, dim).sum(1)   # exact in any order
        assert np.array_equal(out.cpu().numpy(), want)
        assert st["misses"] > 32768 and st["sq_full"] == 0, st
