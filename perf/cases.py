"""Workloads of the scatter/gather engine that its speed is judged by, each through the package's public calls.

A case is a dict of plain values: the application (`op`), the graph (`kind`, `vertices`, `degree`, `partition`) and
the call's options.  Graphs are synthetic and made on the GPU from a seed: R-MAT with a/b/c/d = 0.57/0.19/0.19/0.05
or uniform, self loops and repeated edges removed, as in the benchmark and the report; vertex counts that are no
power of two scale the IDs of the next larger R-MAT."""
from __future__ import annotations

import math

import torch

import paper_1806_08092_gb300 as gp

ROOT_DEGREE = 16  # BFS / SSSP / PPR sources are drawn among vertices with at least this many out-edges


def listed():
    return [
        # a service answering single traversals of a small graph: latency, launches and host round trips
        dict(name="bfs-small", op="bfs", kind="rmat", vertices=1 << 14, degree=16, partition=1024, bw=2),
        # ten PageRank iterations on a graph that stays in L2
        dict(name="pagerank-small", op="pagerank", kind="rmat", vertices=1 << 16, degree=16, partition=1024, iters=10,
             tol=0.0, bf16=False),
        # the headline: PageRank to an L1 change below 1e-9 on a web-like graph of a quarter of a billion edges
        dict(name="pagerank-large", op="pagerank", kind="rmat", vertices=1 << 24, degree=16, partition=16384, iters=300,
             tol=1e-9, bf16=False),
        # PageRank where nearly every edge is its own message (no hubs, r close to 1), ragged last partition
        dict(name="pagerank-uniform", op="pagerank", kind="uniform", vertices=6000011, degree=20, partition=0, iters=10,
             tol=0.0, bf16=False),
        # PageRank with BF16 messages, for rankings that need no more than its three digits
        dict(name="pagerank-bf16", op="pagerank", kind="rmat", vertices=1 << 22, degree=16, partition=16384, iters=30,
             tol=0.0, bf16=True),
        # Graph500-style traversal with parents at full size, at the bandwidth ratio the benchmark uses
        dict(name="bfs-large", op="bfs", kind="rmat", vertices=1 << 24, degree=16, partition=16384, bw=8),
        # shortest paths with integer weights on a road- or cost-annotated graph; default options
        dict(name="sssp", op="sssp", kind="rmat", vertices=1 << 22, degree=16, partition=0, bw=2),
        # connected components of an undirected graph with a ragged vertex count
        dict(name="cc", op="cc", kind="rmat", vertices=3500003, degree=14, partition=8192, bw=2),
        # levels from many sources at once (centralities, landmark distances): two passes of 32
        dict(name="msbfs", op="msbfs", kind="rmat", vertices=1 << 21, degree=16, partition=16384, sources=64, bw=2),
        # one user's personalised PageRank to convergence
        dict(name="ppr", op="ppr", kind="rmat", vertices=1 << 20, degree=16, partition=4096, iters=200, tol=1e-9),
        # personalised PageRank for a batch of users (offline recommendations)
        dict(name="ppr-batch", op="ppr_batch", kind="rmat", vertices=1 << 20, degree=16, partition=1024, sources=48,
             iters=40, tol=0.0),
        # a graph that is loaded, traversed and dropped: the layout build and the first traversal
        dict(name="load-bfs", op="load_bfs", kind="rmat", vertices=1 << 21, degree=16, partition=0, bw=2),
    ]


def _size(rng, lo, hi):
    """A vertex count spread over the logarithm of [lo, hi]: a power of two, or any number."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return 1 << int(round(math.log2(n))) if rng.random() < 0.3 else n | 1


def draw(rng):
    op = rng.choice(["pagerank", "pagerank", "bfs", "bfs", "sssp", "cc", "msbfs", "ppr", "ppr_batch", "load_bfs"])
    kind = rng.choice(["rmat", "rmat", "uniform"])
    top = dict(pagerank=22, bfs=23, sssp=22, cc=21, msbfs=21, ppr=20, ppr_batch=20, load_bfs=21)[op]
    n = _size(rng, 1 << 13, 1 << top)
    c = dict(op=op, kind=kind, vertices=n, degree=rng.randint(6, 24))
    if op == "cc" and kind == "uniform":  # sparse enough for more than one component
        c["degree"] = rng.randint(1, 3)
    parts = [0] + [p for p in (1024, 2048, 4096, 8192, 16384) if n // p <= 4096]
    c["partition"] = 1024 if op == "ppr_batch" else rng.choice(parts)
    if op == "pagerank":
        c.update(iters=rng.randint(5, 40), tol=0.0, bf16=rng.random() < 0.25)
        if rng.random() < 0.3:
            c.update(iters=300, tol=1e-9, bf16=False)
    elif op == "ppr":
        c.update(iters=200, tol=rng.choice([1e-6, 1e-9]))
    elif op == "ppr_batch":
        c.update(sources=rng.randint(1, 48), iters=rng.randint(10, 40), tol=0.0)
    else:
        c["bw"] = rng.choice([2, 8])
        if op == "msbfs":
            c["sources"] = rng.randint(2, 64)
    return c


def _keys(case, gen):
    """The distinct edges of the case's graph as ascending keys source * V + destination, without self loops."""
    n, m = case["vertices"], case["vertices"] * case["degree"]
    if case["kind"] == "uniform":
        src = torch.randint(n, (m,), device="cuda", generator=gen)
        dst = torch.randint(n, (m,), device="cuda", generator=gen)
    else:
        scale = max(1, (n - 1).bit_length())
        src = torch.zeros(m, dtype=torch.int32, device="cuda")
        dst = torch.zeros(m, dtype=torch.int32, device="cuda")
        r = torch.empty(m, device="cuda")
        for _ in range(scale):
            torch.rand(m, out=r, generator=gen)
            src.mul_(2).add_(r >= 0.76)
            dst.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        del r
        src, dst = src.long(), dst.long()
        if n != 1 << scale:
            src.mul_(n).bitwise_right_shift_(scale)
            dst.mul_(n).bitwise_right_shift_(scale)
    keep = src != dst
    key = (src.mul_(n).add_(dst))[keep]
    del src, dst, keep
    key = key.sort().values
    if case["op"] == "cc":  # an undirected graph: both directions
        key = torch.cat([key, key % n * n + key // n]).sort().values
    new = torch.ones(key.numel(), dtype=torch.bool, device="cuda")
    new[1:] = key[1:] != key[:-1]
    return key[new]


def _graph(case, seed):
    """(row_ptr int64, col int32, generator for what is drawn next), on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    key, n = _keys(case, gen), case["vertices"]
    row_ptr = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n)
    return row_ptr, (key % n).int(), gen


def _sources(row_ptr, count, gen):
    """Vertices that reach more than a few others: at least 16 out-edges (or the most there are)."""
    deg = row_ptr[1:] - row_ptr[:-1]
    good = (deg >= min(ROOT_DEGREE, int(deg.max()))).nonzero().flatten()
    return [int(v) for v in good[torch.randint(good.numel(), (count,), device="cuda", generator=gen)].cpu()]


def prepare(case, seed):
    row_ptr, col, gen = _graph(case, seed)
    src = _sources(row_ptr, case.get("sources", 1), gen)
    rp, cl = row_ptr.view(torch.uint64), col.view(torch.uint32)
    if case["op"] == "load_bfs":
        return dict(case=case, row_ptr=rp, col=cl, sources=src)
    w = None
    if case["op"] == "sssp":
        w = torch.randint(1, 256, (col.numel(),), dtype=torch.int32, device="cuda", generator=gen)
    return dict(case=case, graph=gp.Graph.from_csr(rp, cl, w, partition_size=case["partition"]), sources=src)


def _ints(t):
    return t.view(torch.int32)  # a view: the same words under a type that every torch operation takes


def run(state):
    c, src = state["case"], state["sources"]
    if c["op"] == "load_bfs":
        g = gp.Graph.from_csr(state["row_ptr"], state["col"], None, partition_size=c["partition"])
        r = g.run("bfs", source=src[0], bw_ratio=(c["bw"], 1))
        g.close()
        return dict(levels=_ints(r.values), parents=_ints(r.parent))
    g = state["graph"]
    if c["op"] == "pagerank":
        return g.run("pagerank", max_iters=c["iters"], tol=c["tol"], msg_bf16=c["bf16"]).values
    if c["op"] == "ppr":
        return g.run("ppr", source=src[0], max_iters=c["iters"], tol=c["tol"]).values
    if c["op"] == "ppr_batch":
        return g.run_ppr_batch(src, max_iters=c["iters"], tol=c["tol"]).values
    if c["op"] == "msbfs":
        return _ints(g.run_msbfs(src, bw_ratio=(c["bw"], 1)).values)
    if c["op"] == "bfs":
        r = g.run("bfs", source=src[0], bw_ratio=(c["bw"], 1))
        return dict(levels=_ints(r.values), parents=_ints(r.parent))
    if c["op"] == "sssp":
        return _ints(g.run("sssp", source=src[0], bw_ratio=(c["bw"], 1)).values)
    return _ints(g.run("cc", bw_ratio=(c["bw"], 1)).values)


def _rounds(case):
    """Iterations of one pass: as asked for, or what convergence to the case's tolerance typically takes
    (90 for PageRank on R-MAT, 95 for personalised PageRank, both at 1e-9)."""
    if case["tol"] > 0:
        return min(case["iters"], int(round(-10 * math.log10(case["tol"]))))
    return case["iters"]


def work(case):
    """One pass's own bytes: every edge (4 B, 8 B with a weight) and every vertex's value read and written once per
    sweep of a fixed-point iteration, once in all for a traversal, which visits each edge once."""
    v, e, op = case["vertices"], case["vertices"] * case["degree"], case["op"]
    if op in ("pagerank", "ppr"):
        n = _rounds(case)
        return dict(bytes=n * (4.0 * e + 12.0 * v), flops=n * (2.0 * e + 3.0 * v))
    if op == "ppr_batch":
        sweeps, s = math.ceil(case["sources"] / 32) * _rounds(case), case["sources"]
        return dict(bytes=sweeps * (4.0 * e + 4.0 * v) + _rounds(case) * 8.0 * v * s, flops=_rounds(case) * 2.0 * e * s)
    if op == "msbfs":
        return dict(bytes=math.ceil(case["sources"] / 32) * (4.0 * e + 4.0 * v) + 4.0 * v * case["sources"], flops=0)
    if op == "sssp":
        return dict(bytes=8.0 * e + 8.0 * v, flops=0)
    if op == "cc":
        return dict(bytes=8.0 * e + 8.0 * v, flops=0)
    return dict(bytes=4.0 * e + (12.0 if op == "bfs" else 16.0) * v, flops=0)


def exact(case, seed):
    """PageRank and personalised PageRank in 64 bits as repeated sparse products; the other results are whole numbers."""
    if case["op"] not in ("pagerank", "ppr", "ppr_batch"):
        return None
    n = case["vertices"]
    row_ptr, col, gen = _graph(case, seed)
    src = _sources(row_ptr, case.get("sources", 1), gen)
    deg = row_ptr[1:] - row_ptr[:-1]
    of = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    key = (col.long() * n + of).sort().values  # in-edges by destination
    del of
    into = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n)
    a = torch.sparse_csr_tensor(into, key % n, torch.ones(key.numel(), dtype=torch.float64, device="cuda"), (n, n))
    del key
    inv = torch.where(deg > 0, 1.0 / deg.clamp(min=1).double(), 0.0).unsqueeze(1)
    d = 0.85

    def iterate(x, base):
        for i in range(case["iters"]):
            new = base + d * (a @ (x * inv))
            change = (new - x).abs().sum(0).max()
            x = new
            if case["tol"] > 0 and float(change) < case["tol"]:
                break
        return x

    if case["op"] == "pagerank":
        x = torch.full((n, 1), 1.0 / n, dtype=torch.float64, device="cuda")
        return iterate(x, torch.full_like(x, (1 - d) / n)).flatten()
    rows = []
    for b in range(0, len(src), 32):
        part = src[b:b + 32]
        x = torch.zeros((n, len(part)), dtype=torch.float64, device="cuda")
        x[part, range(len(part))] = 1.0
        rows.append(iterate(x, (1 - d) * x).T)
    return rows[0].flatten() if case["op"] == "ppr" else torch.cat(rows).contiguous()
