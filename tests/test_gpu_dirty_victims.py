"""MODIFIED victims claimed by many lanes of a warp at once: each is copied to its staging page by
the whole warp, whose reads follow the claiming lane's fence.  A cache full of MODIFIED lines
(a gradient step on every page) is prefetched over, then every page is read: the bytes are the
oracle's, on reads and on the store, and every dirty epoch was written once."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import PAGE, Ctx, assert_cache_invariants  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("ways,devices", [(8, 1), (8, 2), (4, 1)])
@pytest.mark.parametrize("mode", [ag.AGILE_SYNC, ag.AGILE_ASYNC])
def test_dirty_victims_keep_their_bytes(ways, devices, mode):
    pages, dim, lr = 4096, PAGE // 4, 2.0 ** -4
    T = synth.table_normal(1, pages, dim)
    idx = np.arange(pages, dtype=np.int64)[::-1].copy()
    off = np.arange(pages + 1, dtype=np.int64)
    gout = synth.table_normal(2, pages, dim)
    want = oracle.sgd(T, *oracle.embedding_bag_backward(pages, idx, off, gout), lr)
    d_idx, d_off, d_g = (torch.from_numpy(x).to(DEV) for x in (idx, off, gout))
    order = torch.from_numpy(np.argsort(synth.uniform01(3, pages)).astype(np.int64)).to(DEV)
    with Ctx(T.nbytes, cache_bytes=T.nbytes // 4, ways=ways, num_queues=16, queue_depth=64, num_devices=devices) as c:
        c.put(0, T)
        ag.agile_reset_stats(c.h)
        ag.agile_embedding_bag_backward(c.h, 0, pages, dim, d_idx.data_ptr(), d_off.data_ptr(), pages, pages,
                                        d_g.data_ptr(), lr, 0, mode, c.stream)
        ag.agile_prefetch(c.h, order.data_ptr(), pages, c.stream)
        out = torch.empty((pages, PAGE), dtype=torch.uint8, device=DEV)
        ag.agile_read_async(c.h, order.data_ptr(), pages, out.data_ptr(), 0, mode, c.stream)
        torch.cuda.synchronize()
        c.check()
        assert np.array_equal(out.cpu().numpy(), want.view(np.uint8).reshape(pages, PAGE)[order.cpu().numpy()])
        ag.agile_flush(c.h, c.stream)
        torch.cuda.synchronize()
        c.check()
        assert_cache_invariants(c)
        _, writes, dirtied = ag.agile_page_io(c.h, 0, pages)
        assert np.array_equal(writes, dirtied)
        assert np.array_equal(c.get(0, T.nbytes), want.view(np.uint8).reshape(-1))
