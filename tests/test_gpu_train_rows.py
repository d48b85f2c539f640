"""The backward's row sort and its sums of rows of few and of many positions at the sizes where
they can go wrong (tile and digit edges, segments around the split's length), bit for bit
against the oracle: both add the gradient rows in increasing position, so no tolerance."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import Ctx  # noqa: E402

DEV = "cuda:0"


def _check(rows, dim, idx, n_bags, lr, mode=ag.AGILE_ASYNC):
    n = len(idx)
    off = np.minimum(np.arange(n_bags + 1, dtype=np.int64) * -(-n // n_bags), n)
    T = synth.table_normal(1, rows, dim)
    gout = synth.table_normal(2, n_bags, dim)
    want, touched = oracle.embedding_bag_backward(rows, idx, off, gout)
    d_idx, d_off, d_g = (torch.from_numpy(x).to(DEV) for x in (idx, off, gout))
    with Ctx(T.nbytes, cache_bytes=max(T.nbytes // 4, 64 * 4096), ways=8, num_queues=16, queue_depth=64) as c:
        c.put(0, T)
        for step in (0.0, lr):
            G = torch.full((rows, dim), float("nan"), dtype=torch.float32, device=DEV)
            ag.agile_embedding_bag_backward(c.h, 0, rows, dim, d_idx.data_ptr(), d_off.data_ptr(), n_bags, n,
                                            d_g.data_ptr(), step, G.data_ptr(), mode, c.stream)
            torch.cuda.synchronize()
            c.check()
            assert np.array_equal(G.cpu().numpy().view(np.uint32), want.view(np.uint32))
        ag.agile_flush(c.h, c.stream)
        torch.cuda.synchronize()
        got = c.get(0, T.nbytes).view(np.float32).reshape(rows, dim)
        assert np.array_equal(got.view(np.uint32), oracle.sgd(T, want, touched, lr).view(np.uint32))


@pytest.mark.parametrize("dim", [4, 16, 32, 64, 128, 256, 1024])
def test_segments_around_the_split(dim):
    span = max(64, dim // 4)
    lens = [1, span - 1, span, span + 1, 31, 32, 33, 2 * span, 7 * 32, 4 * 32 + 1, 2, 1000]
    row = np.repeat(np.arange(len(lens)) * 3, lens).astype(np.int64)
    idx = row[np.argsort(synth.uniform01(3, len(row)), kind="stable")]
    _check(3 * len(lens), dim, np.ascontiguousarray(idx), 37, 2.0 ** -5)


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1024, 1025, 5000, (1 << 20) + 1])
@pytest.mark.parametrize("rows", [1, 2, 256, 257, 70_001])
def test_tiles_and_digits(n, rows):
    idx = synth.indices_uniform(4, n, rows)
    idx[0] = rows - 1
    _check(rows, 4, idx, min(n, 301), 2.0 ** -6, ag.AGILE_SYNC if n % 2 else ag.AGILE_ASYNC)


def test_index_out_of_range_is_reported():
    rows, dim = 100, 16
    d_idx = torch.tensor([1, 2, rows, 4], device=DEV)
    d_off = torch.tensor([0, 4], device=DEV)
    g = torch.ones(1, dim, device=DEV)
    G = torch.empty(rows, dim, device=DEV)
    with Ctx(rows * dim * 4, cache_bytes=64 * 4096, ways=8, num_queues=16, queue_depth=64) as c:
        ag.agile_embedding_bag_backward(c.h, 0, rows, dim, d_idx.data_ptr(), d_off.data_ptr(), 1, 4, g.data_ptr(),
                                        0.0, G.data_ptr(), ag.AGILE_SYNC, c.stream)
        torch.cuda.synchronize()
        assert ag.agile_check(c.h) == ag.AGILE_EINVAL
