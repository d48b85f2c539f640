"""Backward + SGD through full queues: misses that claim a line and then find no queue slot give
the line up again, and no page may end with two valid copies (one of them loses updates).
The flushed store equals the oracle's table bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import Ctx, assert_cache_invariants  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("mode,queues,depth", [(ag.AGILE_SYNC, 4, 64), (ag.AGILE_ASYNC, 4, 64),
                                               (ag.AGILE_ASYNC, 128, 256)])
def test_no_update_is_lost_when_queues_are_full(mode, queues, depth):
    rows, dim, n_bags, pool, steps = 1 << 17, 128, 4096, 20, 8
    T = synth.table_normal(1, rows, dim)
    idx = synth.Zipf(rows, 1.1, permute=True, seed=2).rows(3, n_bags * pool)
    off = synth.bags_fixed(n_bags, pool)
    gout = synth.table_normal(4, n_bags, dim)
    lr = 2.0 ** -6
    G, touched = oracle.embedding_bag_backward(rows, idx, off, gout)
    d_idx, d_off, d_g = (torch.from_numpy(x).to(DEV) for x in (idx, off, gout))
    want = T
    with Ctx(T.nbytes, cache_bytes=T.nbytes // 4, ways=8, num_queues=queues, queue_depth=depth) as c:
        c.put(0, T)
        for _ in range(steps):
            want = oracle.sgd(want, G, touched, lr)
            ag.agile_embedding_bag_backward(c.h, 0, rows, dim, d_idx.data_ptr(), d_off.data_ptr(), n_bags, len(idx),
                                            d_g.data_ptr(), lr, 0, mode, c.stream)
            torch.cuda.synchronize()
            c.check()
        assert_cache_invariants(c)
        assert c.stats()["sq_full"] > 0, "the queues were never full"
        ag.agile_flush(c.h, c.stream)
        torch.cuda.synchronize()
        got = c.get(0, T.nbytes).view(np.float32).reshape(rows, dim)
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
