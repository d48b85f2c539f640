"""Performance cases: the calls that a program makes of this library, over their usual range.

Every case is a call (or the few calls of one step) through the public entry points of
``paper_2504_19365_gb300``.  The families:

  bag       sum-pooled embedding-bag lookups through the HBM cache
  pipeline  a batch of lookups over several tables, each followed by a compute phase
  train     forward, backward and SGD step of one batch, the table written back
  bfs       breadth-first search over a CSR graph on the store
  spmv      sparse matrix-vector product over the same layout
  read      pages read from the store into a device buffer
  write     pages written to the store, waited for and read back
  serve     a burst of lookup requests through the resident serving loop

A call repeated on one state finds the cache as the call before it left it, as in a
program that keeps its context: what fits stays resident, what does not is read again.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2504_19365_gb300 as ag
from paper_2504_19365_gb300 import autograd as ag_autograd

PAGE = 4096
FMA_A, FMA_B = 1.0 - 2.0 ** -12, 2.0 ** -10  # the pipeline's compute phase: x = fma(x, FMA_A, FMA_B)
MODES = {"sync": ag.AGILE_SYNC, "async": ag.AGILE_ASYNC}


def listed():
    return [
        # an online lookup of a few users: the table is resident, latency and launches count
        bag("bag_small", rows=4096, dim=64, bags=64, pooling=8, cache=1.5),
        # offline scoring against a resident table: bandwidth of the hit path
        bag("bag_resident", rows=1 << 20, dim=128, bags=65536, pooling=16, cache=1.25),
        # a batch of uniform lookups through a cache of an eighth of the table: misses
        bag("bag_cold", rows=65536, dim=128, bags=256, pooling=16, cache=0.125),
        # a recommendation batch: ragged bags, skewed rows, the blocking mode
        bag("bag_ragged", rows=1_000_003, dim=64, bags=2049, pooling=64, cache=0.2, ragged=True, zipf=1.05,
            mode="sync"),
        # the lookups of eight features with the dense layers' work behind each
        dict(name="pipeline", family="pipeline", tables=8, rows=100_000, dim=64, bags=2048, pooling=32, iters=256,
             cache=0.2, zipf=1.05, mode="async"),
        # one training step of a feature table kept on the store
        dict(name="train_sgd", family="train", rows=1 << 18, dim=128, bags=4096, pooling=20, cache=0.25, zipf=1.1,
             optimizer="sgd", mode="async"),
        # graph traversal with a cache of an eighth of the edges, and of a small graph
        graph("bfs_rmat20", "bfs", scale=20, edge_factor=16, cache=0.125),
        graph("bfs_rmat14", "bfs", scale=14, edge_factor=8, cache=0.5),
        # one product of an iterative solver or of PageRank
        graph("spmv_rmat20", "spmv", scale=20, edge_factor=16, cache=0.125),
        # a restart or a scan: random pages into a device buffer, most of them cold
        dict(name="read_pages", family="read", store_pages=131072, pages=65536, cache=0.125, mode="async"),
        # spilled activations: pages written, waited for and read back
        dict(name="write_pages", family="write", store_pages=32768, pages=8192, cache=0.125, mode="async"),
        # a burst of requests of uneven sizes at a serving process
        dict(name="serve_burst", family="serve", tables=8, rows=100_000, dim=64, requests=48, max_bags=512,
             pooling=64, cache=0.2, zipf=1.05, mode="async"),
    ]


def bag(name, *, rows, dim, bags, pooling, cache, ragged=False, zipf=0.0, mode="async", ways=8, devices=1):
    return dict(name=name, family="bag", rows=rows, dim=dim, bags=bags, pooling=pooling, cache=cache, ragged=ragged,
                zipf=zipf, mode=mode, ways=ways, devices=devices)


def graph(name, family, *, scale, edge_factor, cache, kind="rmat", mode="async"):
    return dict(name=name, family=family, kind=kind, scale=scale, edge_factor=edge_factor, cache=cache, mode=mode)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    mode = rng.choice(["async", "async", "sync"])
    family = rng.choice(["bag", "bag", "bag", "pipeline", "train", "bfs", "bfs", "spmv", "read", "write", "serve"])
    if family == "bag":
        dim = rng.choice([16, 32, 64, 128, 256, 1024])
        rows = log_int(2000, min(1_000_000, (512 << 20) // (4 * dim)))
        resident = rng.random() < 0.5
        pooling = rng.randint(1, 64)
        bags = log_int(16, max(17, min(65536, (1_000_000 if resident else 65_000) * 16 // (pooling * max(16, dim // 8)))))
        case = bag(None, rows=rows, dim=dim, bags=bags, pooling=pooling,
                   cache=1.5 if resident else rng.choice([0.125, 0.2, 0.5]), ragged=rng.random() < 0.5,
                   zipf=rng.choice([0.0, 1.05]), mode=mode, ways=rng.choice([8, 8, 4]),
                   devices=rng.choice([1, 1, 2]))
        del case["name"]
        return case
    if family == "pipeline":
        return dict(family=family, tables=rng.randint(2, 8), rows=log_int(10_000, 100_000), dim=rng.choice([32, 64]),
                    bags=log_int(64, 2000), pooling=rng.randint(1, 32), iters=rng.randint(0, 256),
                    cache=rng.choice([0.2, 0.5]), zipf=1.05, mode=mode)
    if family == "train":
        return dict(family=family, rows=log_int(4000, 260_000), dim=rng.choice([32, 64, 128]), bags=log_int(32, 4000),
                    pooling=rng.randint(1, 20), cache=rng.choice([0.25, 0.5, 1.25]), zipf=rng.choice([0.0, 1.1]),
                    optimizer=rng.choice(["sgd", "table"]), mode=mode)
    if family in ("bfs", "spmv"):
        case = graph(None, family, scale=rng.randint(10, 19), edge_factor=rng.randint(4, 16),
                     cache=rng.choice([0.125, 0.25, 1.25]), kind=rng.choice(["rmat", "rmat", "uniform"]), mode=mode)
        del case["name"]
        return case
    if family == "read":
        return dict(family=family, store_pages=log_int(4096, 131_000), pages=log_int(1, 60_000),
                    cache=rng.choice([0.125, 0.5]), mode=mode)
    if family == "write":
        return dict(family=family, store_pages=log_int(8192, 32_000), pages=log_int(1, 8000),
                    cache=rng.choice([0.125, 0.5]), mode=mode)
    return dict(family="serve", tables=rng.randint(1, 8), rows=log_int(10_000, 100_000), dim=rng.choice([32, 64, 128]),
                requests=rng.randint(1, 48), max_bags=log_int(8, 400), pooling=rng.randint(1, 64), cache=0.2,
                zipf=1.05, mode=mode)


# ----------------------------------------------------------------------------- inputs

def generator(seed, stream=0):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + stream)


def indices(g, n, rows, zipf):
    """n rows, uniform or Zipf(zipf) by rank with the hot rows spread over the table."""
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    if not zipf:
        return (u * rows).long().clamp_(max=rows - 1)
    cdf = torch.arange(1, rows + 1, device="cuda", dtype=torch.float64).pow_(-zipf).cumsum(0)
    rank = torch.searchsorted(cdf, u * cdf[-1]).clamp_(max=rows - 1)
    step = max(1, 0x9E3779B1 % rows)
    while math.gcd(step, rows) != 1:
        step += 1
    return rank * step % rows


def bag_offsets(g, bags, pooling, ragged):
    off = torch.arange(bags + 1, device="cuda", dtype=torch.int64)
    if not ragged:
        return off * pooling
    off[0] = 0
    off[1:] = torch.randint(1, pooling + 1, (bags,), generator=g, device="cuda").cumsum(0)
    return off


def table_values(g, rows, dim):
    return torch.randn(rows, dim, generator=g, device="cuda")


def csr(case, seed):
    """int64 offsets, int32 sorted columns of a symmetric graph without loops or duplicates."""
    g = generator(seed)
    n, m = 1 << case["scale"], case["edge_factor"] << case["scale"]
    if case["kind"] == "uniform":
        src, dst = (torch.randint(0, n, (m,), generator=g, device="cuda") for _ in range(2))
    else:  # R-MAT, (a, b, c) = (0.57, 0.19, 0.19)
        src, dst = (torch.zeros(m, device="cuda", dtype=torch.int64) for _ in range(2))
        for _ in range(case["scale"]):
            u = torch.rand(m, generator=g, device="cuda")
            src = 2 * src + (u >= 0.76)
            dst = 2 * dst + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    key = torch.cat([src * n + dst, dst * n + src])[torch.cat([src != dst, src != dst])]
    key = torch.unique(key)
    off = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
    off[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return n, off, (key % n).int()


def serve_requests(case, seed):
    """(table, offsets, indices) of each request: bags spread evenly over their logarithm, pooling uniform."""
    rng = np.random.RandomState(int(seed) % (1 << 32))
    g = generator(seed, 1)
    reqs = []
    for i in range(case["requests"]):
        bags = int(round(case["max_bags"] ** ((i + 0.5) * 0.6180339887498949 % 1)))
        off = bag_offsets(g, bags, int(rng.randint(1, case["pooling"] + 1)), False)
        reqs.append((int(rng.randint(case["tables"])), off, indices(g, int(off[-1]), case["rows"], case["zipf"])))
    return reqs


# ----------------------------------------------------------------------------- library state

def round_up(n, unit=PAGE):
    return (int(n) + unit - 1) // unit * unit


class Context:
    """A library context with its store filled from tensors, each at a page boundary."""

    def __init__(self, arrays, cache_bytes, ways=8, devices=1):
        self.at, size = [], 0
        for a in arrays:
            self.at.append(size)
            size += round_up(a.numel() * a.element_size())
        cache = max(round_up(cache_bytes, ways * PAGE), 64 * ways * PAGE)
        cfg = ag.agile_config_default(store_bytes=size, cache_bytes=cache, ways=ways, num_devices=devices)
        self.handle = ag.agile_init(cfg)
        self.pages = size // PAGE
        for off, a in zip(self.at, arrays):
            host = a.cpu().numpy()
            ag.agile_store_write(self.handle, off, host.ctypes.data, host.nbytes)

    def warm(self):
        """Bring the whole store into the cache (a cache that holds it)."""
        pages = torch.arange(self.pages, device="cuda", dtype=torch.int64)
        ag.agile_prefetch(self.handle, pages.data_ptr(), self.pages, stream())
        torch.cuda.synchronize()

    def __del__(self):
        if getattr(self, "handle", None) and ag is not None:
            handle, self.handle = self.handle, None
            ag.agile_destroy(handle)


def stream():
    return torch.cuda.current_stream().cuda_stream


def cache_of(case, nbytes):
    return int(case["cache"] * nbytes)


def prepare(case, seed):
    case = dict(case)
    return case, PREPARE[case["family"]](case, seed)


def prepare_bag(case, seed):
    g = generator(seed)
    table = table_values(g, case["rows"], case["dim"])
    off = bag_offsets(g, case["bags"], case["pooling"], case["ragged"])
    idx = indices(g, int(off[-1]), case["rows"], case["zipf"])
    ctx = Context([table], cache_of(case, table.numel() * 4), case["ways"], case["devices"])
    if case["cache"] >= 1:
        ctx.warm()
    return ctx, idx, off, torch.empty(case["bags"], case["dim"], device="cuda")


def run_bag(case, s):
    ctx, idx, off, out = s
    ag.agile_embedding_bag(ctx.handle, 0, case["rows"], case["dim"], idx.data_ptr(), off.data_ptr(), case["bags"],
                           out.data_ptr(), MODES[case["mode"]], stream())
    return out


def pipeline_inputs(case, seed):
    g = generator(seed)
    tables = [table_values(g, case["rows"], case["dim"]) for _ in range(case["tables"])]
    idx = indices(g, case["tables"] * case["bags"] * case["pooling"], case["rows"], case["zipf"])
    return tables, idx


def prepare_pipeline(case, seed):
    tables, idx = pipeline_inputs(case, seed)
    ctx = Context(tables, cache_of(case, len(tables) * tables[0].numel() * 4))
    return ctx, idx, torch.empty(case["bags"], case["tables"] * case["dim"], device="cuda")


def run_pipeline(case, s):
    ctx, idx, out = s
    ag.agile_embedding_pipeline(ctx.handle, 0, round_up(case["rows"] * case["dim"] * 4), case["tables"], case["rows"],
                                case["dim"], idx.data_ptr(), case["pooling"], case["bags"], 1, case["iters"],
                                out.data_ptr(), MODES[case["mode"]], stream())
    return out


LEARNING_RATE = 2.0 ** -6


def train_inputs(case, seed):
    g = generator(seed)
    table = table_values(g, case["rows"], case["dim"])
    off = bag_offsets(g, case["bags"], case["pooling"], False)
    idx = indices(g, int(off[-1]), case["rows"], case["zipf"])
    grad = torch.randn(case["bags"], case["dim"], generator=g, device="cuda")
    return table, off, idx, grad


def prepare_train(case, seed):
    table, off, idx, grad = train_inputs(case, seed)
    ctx = Context([table], cache_of(case, table.numel() * 4))
    one = torch.arange(idx.numel() + 1, device="cuda", dtype=torch.int64)
    after = torch.empty(table.shape if case["optimizer"] == "table" else (idx.numel(), case["dim"]), device="cuda")
    return ctx, off, idx, grad, one, after


def run_train(case, s):
    ctx, off, idx, grad, one, after = s
    mode = MODES[case["mode"]]
    sgd = case["optimizer"] == "sgd"
    out = ag_autograd.cached_embedding_bag(ctx.handle, 0, case["rows"], case["dim"], idx, off, LEARNING_RATE, mode)
    if sgd:
        # the fused SGD step: changed pages are written back, the batch's new rows are looked up
        out.backward(grad)
        ag.agile_flush(ctx.handle, stream())
        ag.agile_embedding_bag(ctx.handle, 0, case["rows"], case["dim"], idx.data_ptr(), one.data_ptr(),
                               idx.numel(), after.data_ptr(), mode, stream())
    else:
        # the gradient of the whole table, for an optimizer of the program's own
        ag.agile_embedding_bag_backward(ctx.handle, 0, case["rows"], case["dim"], idx.data_ptr(), off.data_ptr(),
                                        case["bags"], idx.numel(), grad.data_ptr(), 0.0, after.data_ptr(), mode,
                                        stream())
    return {"pooled": out.detach(), "rows" if sgd else "gradient": after}


def prepare_bfs(case, seed):
    n, off, cols = csr(case, seed)
    # an edge's end: a vertex of the graph's large component in all but a few draws
    at = int(torch.randint(0, cols.numel(), (1,), generator=generator(seed, 1), device="cuda"))
    ctx = Context([off, cols], cache_of(case, cols.numel() * 4))
    return ctx, n, int(cols[at]), torch.empty(n, device="cuda", dtype=torch.int32), torch.zeros(
        1, device="cuda", dtype=torch.int64)


def run_bfs(case, s):
    ctx, n, source, level, scanned = s
    ag.agile_bfs(ctx.handle, ctx.at[0], ctx.at[1], n, source, level.data_ptr(), scanned.data_ptr(),
                 MODES[case["mode"]], stream())
    return level, scanned


def spmv_inputs(case, seed):
    n, off, cols = csr(case, seed)
    g = generator(seed, 1)
    return n, off, cols, torch.randn(cols.numel(), generator=g, device="cuda"), torch.randn(n, generator=g, device="cuda")


def prepare_spmv(case, seed):
    n, off, cols, vals, x = spmv_inputs(case, seed)
    ctx = Context([off, cols, vals], cache_of(case, cols.numel() * 8))
    return ctx, n, x, torch.empty(n, device="cuda")


def run_spmv(case, s):
    ctx, n, x, y = s
    ag.agile_spmv(ctx.handle, *ctx.at, n, n, x.data_ptr(), y.data_ptr(), 0, MODES[case["mode"]], stream())
    return y


def store_words(case, seed):
    return torch.randint(-2 ** 31, 2 ** 31, (case["store_pages"], PAGE // 4), generator=generator(seed),
                         device="cuda", dtype=torch.int32)


def prepare_pages(case, seed):
    words = store_words(case, seed)
    ctx = Context([words], cache_of(case, words.numel() * 4))
    g = generator(seed, 1)
    n = case["pages"]
    if case["family"] == "read":
        pages = torch.randint(0, case["store_pages"], (n,), generator=g, device="cuda")
    else:  # every page of a spill is another one
        pages = torch.randperm(case["store_pages"], generator=g, device="cuda")[:n].contiguous()
    src = torch.randint(-2 ** 31, 2 ** 31, (n, PAGE // 4), generator=g, device="cuda", dtype=torch.int32)
    tokens = torch.empty(n, device="cuda", dtype=torch.int64)
    status = torch.empty(n, device="cuda", dtype=torch.int32)
    return ctx, pages, src, tokens, status, torch.empty_like(src)


def run_read(case, s):
    ctx, pages, _, tokens, status, dst = s
    n = case["pages"]
    ag.agile_read_async(ctx.handle, pages.data_ptr(), n, dst.data_ptr(), tokens.data_ptr(), MODES[case["mode"]],
                        stream())
    ag.agile_wait(ctx.handle, tokens.data_ptr(), n, status.data_ptr(), stream())
    return dst, status


def run_write(case, s):
    ctx, pages, src, tokens, status, dst = s
    n = case["pages"]
    ag.agile_write_async(ctx.handle, pages.data_ptr(), n, src.data_ptr(), tokens.data_ptr(), stream())
    ag.agile_wait(ctx.handle, tokens.data_ptr(), n, status.data_ptr(), stream())
    ag.agile_read_async(ctx.handle, pages.data_ptr(), n, dst.data_ptr(), 0, MODES[case["mode"]], stream())
    return dst, status


def serve_tables(case, seed):
    g = generator(seed)
    return [table_values(g, case["rows"], case["dim"]) for _ in range(case["tables"])]


def prepare_serve(case, seed):
    tables = serve_tables(case, seed)
    ctx = Context(tables, cache_of(case, len(tables) * tables[0].numel() * 4))
    reqs = serve_requests(case, seed)
    out = torch.empty(sum(off.numel() - 1 for _, off, _ in reqs), case["dim"], device="cuda")
    calls, at = [], 0
    for k, off, idx in reqs:
        bags = off.numel() - 1
        calls.append(ag.agile_lookup_req(ctx.at[k], case["rows"], case["dim"], idx.data_ptr(), off.data_ptr(), bags,
                                         out[at].data_ptr()))
        at += bags
    return ctx, reqs, calls, np.zeros(len(calls), np.uint64), np.zeros(len(calls), np.uint64), out


def run_serve(case, s):
    ctx, _, calls, arrival, latency, out = s
    ag.agile_serve_replay(ctx.handle, calls, arrival.ctypes.data_as(ctypes.c_void_p),
                          latency.ctypes.data_as(ctypes.c_void_p), MODES[case["mode"]], stream())
    return out


PREPARE = {"bag": prepare_bag, "pipeline": prepare_pipeline, "train": prepare_train, "bfs": prepare_bfs,
           "spmv": prepare_spmv, "read": prepare_pages, "write": prepare_pages, "serve": prepare_serve}
RUN = {"bag": run_bag, "pipeline": run_pipeline, "train": run_train, "bfs": run_bfs, "spmv": run_spmv,
       "read": run_read, "write": run_write, "serve": run_serve}


def run(state):
    case, s = state
    return RUN[case["family"]](case, s)


# ----------------------------------------------------------------------------- what a call cannot do without

def lookups(case):
    return case["bags"] * (case["pooling"] + 1) / 2 if case.get("ragged") else case["bags"] * case["pooling"]


def work(case):
    """Bytes: each looked-up row or scanned entry once, its index, and the outputs.  Flops: adds and multiplies."""
    f = case["family"]
    if f == "bag":
        n, dim = lookups(case), case["dim"]
        return {"bytes": n * (4 * dim + 8) + case["bags"] * (4 * dim + 8), "flops": n * dim}
    if f == "pipeline":
        pooled = case["tables"] * case["bags"]
        n, dim = pooled * case["pooling"], case["dim"]
        return {"bytes": n * (4 * dim + 8) + pooled * 4 * dim, "flops": n * dim + 2 * pooled * dim * case["iters"]}
    if f == "train":
        # forward rows, gradient rows, and the touched rows changed and looked up (or the gradient written)
        n, dim = lookups(case), case["dim"]
        touched = case["rows"] * (1 - math.exp(-n / case["rows"])) if not case["zipf"] else min(case["rows"], n) / 3
        last = (8 * touched + 4 * n) * dim if case["optimizer"] == "sgd" else 4 * case["rows"] * dim
        return {"bytes": n * (4 * dim + 16) + case["bags"] * 8 * dim + last, "flops": 2 * n * dim + 2 * touched * dim}
    if f in ("bfs", "spmv"):
        n, entries = 1 << case["scale"], 2 * case["edge_factor"] << case["scale"]
        if f == "bfs":
            return {"bytes": 4 * entries + 12 * n, "flops": 0}
        return {"bytes": 8 * entries + 16 * n, "flops": 2 * entries}
    if f == "read":
        return {"bytes": case["pages"] * (2 * PAGE + 8), "flops": 0}
    if f == "write":
        return {"bytes": case["pages"] * (4 * PAGE + 8), "flops": 0}
    bags = (case["max_bags"] - 1) / math.log(case["max_bags"]) * case["requests"]
    n, dim = bags * (case["pooling"] + 1) / 2, case["dim"]
    return {"bytes": n * (4 * dim + 8) + bags * 4 * dim, "flops": n * dim}


# ----------------------------------------------------------------------------- the results in 64 bits

def pooled64(table, off, idx):
    """Sum-pooled rows in float64, a slice of the bags at a time."""
    out = torch.zeros(off.numel() - 1, table.shape[1], device="cuda", dtype=torch.float64)
    bag_of = torch.repeat_interleave(torch.arange(out.shape[0], device="cuda"), off[1:] - off[:-1])
    step = max(1, (1 << 27) // table.shape[1])
    for i in range(0, idx.numel(), step):
        out.index_add_(0, bag_of[i:i + step], table[idx[i:i + step]].double())
    return out


def exact_bag(case, seed):
    g = generator(seed)
    table = table_values(g, case["rows"], case["dim"])
    off = bag_offsets(g, case["bags"], case["pooling"], case["ragged"])
    return pooled64(table, off, indices(g, int(off[-1]), case["rows"], case["zipf"]))


def exact_pipeline(case, seed):
    tables, idx = pipeline_inputs(case, seed)
    idx = idx.view(case["tables"], case["bags"], case["pooling"])
    out = torch.cat([t[i].double().sum(1) for t, i in zip(tables, idx)], 1)
    for _ in range(case["iters"]):
        out = out * FMA_A + FMA_B
    return out


def exact_train(case, seed):
    table, off, idx, grad = train_inputs(case, seed)
    pooled = pooled64(table, off, idx)
    gradient = torch.zeros(table.shape, device="cuda", dtype=torch.float64)
    bag_of = torch.repeat_interleave(torch.arange(case["bags"], device="cuda"), off[1:] - off[:-1])
    gradient.index_add_(0, idx, grad.double()[bag_of])
    if case["optimizer"] == "table":
        return {"pooled": pooled, "gradient": gradient}
    return {"pooled": pooled, "rows": (table.double() - LEARNING_RATE * gradient)[idx]}


def exact_spmv(case, seed):
    n, off, cols, vals, x = spmv_inputs(case, seed)
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    return torch.zeros(n, device="cuda", dtype=torch.float64).index_add_(0, row, vals.double() * x.double()[cols.long()])


def exact_serve(case, seed):
    tables = serve_tables(case, seed)
    return torch.cat([pooled64(tables[k], off, idx) for k, off, idx in serve_requests(case, seed)])


def exact(case, seed):
    """What ``run`` returns on a new state; None where every output is a whole number or bytes."""
    f = {"bag": exact_bag, "pipeline": exact_pipeline, "train": exact_train, "spmv": exact_spmv,
         "serve": exact_serve}.get(case["family"])
    return f(case, seed) if f else None
