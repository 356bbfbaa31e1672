"""The PC gather's destination runs at the edges of their classes, rows and weight formats, against the oracle.

The entries of one destination in a block are stored by length: single entries, 2-3, 4-7, and pieces of 7 entries of
longer runs, in rows of 64 pieces whose lanes hold one or two.  Lengths on both sides of every such edge, alone and
among others, with repeated edges; column-major bins of every length modulo 8; edge weights on both sides of 16 bits."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGE_LENGTHS = [1, 2, 3, 4, 7, 8, 14, 15, 7 * 31, 7 * 32, 7 * 32 + 1, 7 * 33, 7 * 63, 7 * 64, 7 * 64 + 1, 7 * 65, 7 * 96, 3000]


@pytest.fixture(scope="module", autouse=True)
def lib():
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    return gp


def runs_graph(lengths, n, seed, weight_bits, repeat=False):
    """Vertex 0 reaches every source; destination j * 3 has in-degree lengths[j] (+ a few from vertex 0's ring)."""
    rng = np.random.default_rng(seed)
    nsrc = max(max(lengths), 64)
    src0 = 4096  # sources lie in other partitions than the destinations
    u, v = [np.zeros(nsrc, np.int64)], [np.arange(src0, src0 + nsrc)]
    for j, L in enumerate(lengths):
        s = rng.choice(nsrc, L, replace=False) + src0
        if repeat and L > 2:
            s[: L // 2] = s[L // 2: 2 * (L // 2)]  # parallel edges
        u.append(s)
        v.append(np.full(L, (3 * j) % src0))
    u, v = np.concatenate(u), np.concatenate(v)
    g = gg.multigraph(n, u.tolist(), v.tolist())
    w = rng.integers(0, 1 << weight_bits, g.num_edges).astype(np.int32)
    w[0] = (1 << weight_bits) - 1
    g.weights = w
    return g


def check(g, P):
    import paper_1806_08092_gb300 as gp
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=P)
    # a value is a sum of positive FP32 terms in at most three roundings per level: far below 1e-5
    ref, _, _ = O.pagerank(g, 0.85, max_iters=3)
    for mode in ("force_pc", "analytic"):
        x = G.run("pagerank", max_iters=3, mode=mode).values.cpu().numpy().astype(np.float64)
        assert np.max(np.abs(x - ref) / ref) <= 1e-5, mode
    # BF16 messages (relative rounding 2^-9 per message and iteration, three iterations)
    x = G.run("pagerank", max_iters=3, mode="force_pc", msg_bf16=True).values.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(x - ref) / ref) <= 3 * 2.0 ** -8
    level, parent = O.bfs(g, 0)
    r = G.run("bfs", source=0, mode="force_pc")
    assert np.array_equal(r.values.cpu().numpy(), level) and np.array_equal(r.parent.cpu().numpy(), parent)
    dist = O.sssp(g, 0)
    d32 = dist.copy()
    d32[dist == O.U64_INF] = O.U32_INF
    assert np.array_equal(G.run("sssp", source=0, mode="force_pc").values.cpu().numpy(), d32.astype(np.uint32))
    src = [0, 4096, 4097, 5000]
    assert np.array_equal(G.run_msbfs(src, mode="force_pc").values.cpu().numpy(), O.msbfs(g, src))
    if P <= 1024:
        rows = G.run_ppr_batch(src, max_iters=4).values.cpu().numpy().astype(np.float64)
        for row, s in zip(rows, src):
            x, _, _ = O.ppr(g, s, 0.15, max_iters=4)
            assert np.max(np.abs(row - x)) <= 1e-6 * max(np.max(x), 1e-3)
    G.close()


@pytest.mark.parametrize("bits", [16, 17, 28])  # 65535 is the largest weight of the 16-bit format
@pytest.mark.parametrize("P", [32, 1024, 16384])
def test_every_length_together(P, bits):
    check(runs_graph(EDGE_LENGTHS + [1, 2, 5, 9, 1, 3, 30, 1], 9001, 7 * P + bits, bits), P)


@pytest.mark.parametrize("length", EDGE_LENGTHS)
def test_one_length(length):
    check(runs_graph([length], 9001, length, 8), 1024)


@pytest.mark.parametrize("count", [3, 31, 33, 64, 65, 127, 129, 300])
def test_many_runs_of_a_class(count):
    for length in (1, 3, 6, 20):
        check(runs_graph([length] * count, 9001, count, 8), 512)


def test_repeated_edges():
    check(runs_graph(EDGE_LENGTHS, 9001, 3, 17, repeat=True), 1024)


@pytest.mark.parametrize("bits", [8, 20])
def test_rows_in_any_order_give_the_same_graph(bits):
    # the build sorts the rows only when one is out of order; repeated edges with different weights among them
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(12)
    rng = np.random.default_rng(bits)
    u = np.repeat(np.arange(g.num_vertices), np.diff(g.row_ptr.astype(np.int64)))
    u, v = np.concatenate([u, u[:500]]), np.concatenate([g.col.astype(np.int64), g.col[:500].astype(np.int64)])
    w = rng.integers(1, 1 << bits, u.size).astype(np.int32)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=g.num_vertices))]).astype(np.uint64)
    inorder, shuffled = np.lexsort((v, u)), np.lexsort((rng.permutation(u.size), u))
    out = []
    for o in (inorder, shuffled):
        G = gp.Graph.from_csr(row_ptr, v[o].astype(np.uint32), w[o], partition_size=256)
        out.append([G.run(a, source=3, mode=m).values.cpu().numpy() for a in ("bfs", "sssp") for m in ("force_pc", "force_sc")])
        G.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))
