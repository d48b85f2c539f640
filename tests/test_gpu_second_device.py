"""A context on a second device: SpMV, whose kernel needs more dynamic shared memory than a kernel has
without asking, runs on it after it has run on the first one."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import Ctx, round_page  # noqa: E402


def test_spmv_on_every_device():
    if torch.cuda.device_count() < 2:
        pytest.skip("one device")
    n, off, cols = synth.rmat_csr(3, 10, 8)
    vals, x = synth.normal(1, cols.size).astype(np.float32), synth.normal(2, n).astype(np.float32)
    col0 = round_page(off.nbytes)
    val0 = col0 + round_page(cols.nbytes)
    want = oracle.spmv(off, cols, vals, x)
    for dev in range(2):
        with torch.cuda.device(dev), Ctx(val0 + vals.nbytes, cache_bytes=256 << 10, ways=8, num_queues=16,
                                         queue_depth=64, device=dev) as c:
            c.put(0, off)
            c.put(col0, cols)
            c.put(val0, vals)
            d_x, d_y = torch.from_numpy(x).cuda(dev), torch.empty(n, device=f"cuda:{dev}")
            ag.agile_spmv(c.h, 0, col0, val0, n, n, d_x.data_ptr(), d_y.data_ptr(), 0, ag.AGILE_ASYNC, c.stream)
            torch.cuda.synchronize()
            c.check()
            assert np.array_equal(d_y.cpu().numpy().view(np.uint32), want.view(np.uint32))
