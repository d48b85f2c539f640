"""Training steps one after the other on one context (lookup, backward with the fused SGD update,
flush, lookup of the batch's rows): every output of every step equals the oracle's FP32 result
bit for bit, so an update lost in one step would show in the next."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from paper_2504_19365_gb300.autograd import cached_embedding_bag  # noqa: E402
from gpu_util import Ctx, assert_cache_invariants  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("mode", [ag.AGILE_SYNC, ag.AGILE_ASYNC])
@pytest.mark.parametrize("seed", [1, 2])
def test_outputs_of_every_step(mode, seed):
    rows, dim, n_bags, pool, steps, lr = 1 << 16, 128, 4096, 20, 6, 2.0 ** -6
    T = synth.table_normal(10 * seed, rows, dim)
    idx = synth.Zipf(rows, 1.1, permute=True, seed=10 * seed + 1).rows(10 * seed + 2, n_bags * pool)
    off = synth.bags_fixed(n_bags, pool)
    gout = synth.table_normal(10 * seed + 3, n_bags, dim)
    G, touched = oracle.embedding_bag_backward(rows, idx, off, gout)
    d_idx, d_off, d_g = (torch.from_numpy(x).to(DEV) for x in (idx, off, gout))
    one = torch.arange(len(idx) + 1, device=DEV, dtype=torch.int64)
    after = torch.empty((len(idx), dim), dtype=torch.float32, device=DEV)
    want = T
    with Ctx(T.nbytes, cache_bytes=T.nbytes // 4, ways=8) as c:
        c.put(0, T)
        for step in range(steps):
            out = cached_embedding_bag(c.h, 0, rows, dim, d_idx, d_off, lr, mode)
            out.backward(d_g)
            ag.agile_flush(c.h, c.stream)
            ag.agile_embedding_bag(c.h, 0, rows, dim, d_idx.data_ptr(), one.data_ptr(), len(idx), after.data_ptr(),
                                   mode, c.stream)
            torch.cuda.synchronize()
            c.check()
            pooled = oracle.embedding_bag(want, idx, off)
            want = oracle.sgd(want, G, touched, lr)
            assert np.array_equal(out.detach().cpu().numpy().view(np.uint32), pooled.view(np.uint32)), step
            assert np.array_equal(after.cpu().numpy().view(np.uint32), want[idx].view(np.uint32)), step
        assert_cache_invariants(c)
