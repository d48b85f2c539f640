"""The applications at every shape of an engine launch: few CTAs (a service warp in each), many
(service CTAs), and numbers of application warps that leave CTAs unevenly filled.  BFS with long
lists (slice queue, grid barrier, its end watched by one warp a CTA), SpMV with long rows
(shared memory of each warp, carried sums) and the embedding bag, bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2504_19365_gb300 as ag  # noqa: E402
from gpu_util import PAGE, Ctx, assert_cache_invariants, round_page  # noqa: E402

DEV = "cuda:0"


def _graph():
    """Lists of 0 to 40 entries, and some of 255 to 7,000 (around the split into slices)."""
    n = 7001
    deg = synth.uniform_int(1, n, 41)
    deg[synth.uniform_int(2, 12, n)] = [255, 256, 257, 1023, 1024, 1025, 2047, 2048, 2304, 4096, 5000, 7000]
    off = np.zeros(n + 1, dtype=np.int64)
    off[1:] = np.cumsum(deg)
    cols = synth.uniform_int(3, int(off[-1]), n).astype(np.int32)
    return n, off, cols


@pytest.mark.parametrize("max_ctas,app_warps", [(1, 0), (2, 0), (7, 0), (8, 0), (9, 0), (2, 3), (7, 8), (9, 10), (30, 27),
                                                (0, 1), (0, 3), (0, 129), (0, 0)])
@pytest.mark.parametrize("mode", [ag.AGILE_SYNC, ag.AGILE_ASYNC])
def test_every_application(max_ctas, app_warps, mode):
    n, off, cols = _graph()
    vals, x = synth.normal(4, cols.size).astype(np.float32), synth.normal(5, n).astype(np.float32)
    rows, dim = 2000, 64
    T = synth.table_normal(6, rows, dim)
    idx, bag_off = synth.indices_uniform(7, 300 * 11, rows), synth.bags_fixed(300, 11)
    at = np.cumsum([0] + [round_page(a.nbytes) for a in (off, cols, vals, T)])
    with Ctx(int(at[-1]), cache_bytes=128 * PAGE, ways=8, num_queues=16, queue_depth=64, max_ctas=max_ctas,
             wait_timeout_ns=20_000_000_000) as c:
        for a, p in zip((off, cols, vals, T), at):
            c.put(int(p), a)
        ag.agile_config_parallelism(c.h, app_warps)
        level = torch.empty(n, dtype=torch.int32, device=DEV)
        edges = torch.zeros(1, dtype=torch.int64, device=DEV)
        src = int(synth.uniform_int(2, 12, n)[3])
        ag.agile_bfs(c.h, 0, int(at[1]), n, src, level.data_ptr(), edges.data_ptr(), mode, c.stream)
        d_x, y = torch.from_numpy(x).to(DEV), torch.empty(n, device=DEV)
        ag.agile_spmv(c.h, 0, int(at[1]), int(at[2]), n, n, d_x.data_ptr(), y.data_ptr(), 0, mode, c.stream)
        d_idx, d_off = torch.from_numpy(idx).to(DEV), torch.from_numpy(bag_off).to(DEV)
        out = torch.empty((300, dim), device=DEV)
        ag.agile_embedding_bag(c.h, int(at[3]), rows, dim, d_idx.data_ptr(), d_off.data_ptr(), 300, out.data_ptr(),
                               mode, c.stream)
        torch.cuda.synchronize()
        c.check()
        want, scanned = oracle.bfs(off, cols, src)
        assert np.array_equal(level.cpu().numpy(), want) and int(edges.item()) == scanned
        assert np.array_equal(y.cpu().numpy().view(np.uint32), oracle.spmv(off, cols, vals, x).view(np.uint32))
        assert np.array_equal(out.cpu().numpy().view(np.uint32), oracle.embedding_bag(T, idx, bag_off).view(np.uint32))
        assert_cache_invariants(c)
