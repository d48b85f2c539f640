"""Every shape of an engine launch moves pages intact: launches of a few CTAs (a service warp in
each) and of many (service CTAs), one poller for several queues, queues of the smallest
depth, sets of 8 ways and others, several devices, both victim policies.  Pages are
written, read back through a cache of a few lines and compared byte for byte."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import PAGE, Ctx, assert_cache_invariants  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("ctas,queues,depth,ways,devices,policy", [
    (1, 1, 64, 8, 1, 0), (2, 40, 64, 4, 1, 0), (7, 6, 64, 8, 3, 1), (8, 48, 64, 8, 1, 0), (9, 33, 128, 3, 1, 1),
    (30, 5, 64, 8, 5, 0), (0, 1, 64, 8, 1, 0), (0, 300, 64, 8, 2, 1), (0, 1025, 64, 16, 1, 0)])
@pytest.mark.parametrize("mode", [ag.AGILE_SYNC, ag.AGILE_ASYNC])
def test_pages_survive(ctas, queues, depth, ways, devices, policy, mode):
    npages, n = 4099, 3001
    store = synth.uniform_int(1, npages * PAGE // 8, 1 << 62).view(np.uint8)
    pages = np.argsort(synth.uniform01(2, npages))[:n].astype(np.int64)
    new = synth.uniform_int(3, n * PAGE // 8, 1 << 62).view(np.uint8).reshape(n, PAGE)
    with Ctx(npages * PAGE, cache_bytes=12 * ways * PAGE, ways=ways, num_queues=queues, queue_depth=depth,
             num_devices=devices, cache_policy=policy, max_ctas=ctas, wait_timeout_ns=20_000_000_000) as c:
        c.put(0, store)
        d_pages, d_new = torch.from_numpy(pages).to(DEV), torch.from_numpy(new).to(DEV)
        tok = torch.empty(n, dtype=torch.int64, device=DEV)
        status = torch.full((n,), 7, dtype=torch.int32, device=DEV)
        ag.agile_write_async(c.h, d_pages.data_ptr(), n, d_new.data_ptr(), tok.data_ptr(), c.stream)
        ag.agile_wait(c.h, tok.data_ptr(), n, status.data_ptr(), c.stream)
        every = torch.arange(npages, device=DEV).flip(0).contiguous()
        out = torch.empty((npages, PAGE), dtype=torch.uint8, device=DEV)
        ag.agile_read_async(c.h, every.data_ptr(), npages, out.data_ptr(), 0, mode, c.stream)
        torch.cuda.synchronize()
        c.check()
        assert (status == 0).all()
        want = store.reshape(npages, PAGE).copy()
        want[pages] = new
        assert np.array_equal(out.flip(0).cpu().numpy(), want)
        ag.agile_flush(c.h, c.stream)
        torch.cuda.synchronize()
        assert_cache_invariants(c)
        assert np.array_equal(c.get(0, npages * PAGE).reshape(npages, PAGE), want)
