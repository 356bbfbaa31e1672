"""The iteration's kernels on small graphs, which by default run in one launch: with their launches counted, and with
iterations launched ahead of the plan, against the oracle."""
import ctypes

import numpy as np
import pytest

import graphgen as gg
import oracle as O
from test_gpu_runs import EDGE_LENGTHS, runs_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SC_SCATTER, TASK_GATHER, PC_GATHER, MERGE = 2, 3, 4, 5  # kinds of kernel_launches


@pytest.fixture(scope="module", autouse=True)
def lib():
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    return gp


def distances(g, root):
    d = O.sssp(g, root)
    return np.where(d == O.U64_INF, O.U32_INF, d).astype(np.uint32)


@pytest.mark.parametrize("P,bits", [(32, 17), (1024, 16), (16384, 28)])
def test_run_classes_through_the_pc_gather(P, bits):
    # 16- and 32-bit weights, every class and row edge, by kernels that report their launches
    import paper_1806_08092_gb300 as gp
    g = runs_graph(EDGE_LENGTHS + [1, 2, 5, 9, 1, 3, 30, 1], 9001, 7 * P + bits, bits)
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=P)
    ref, _, _ = O.pagerank(g, 0.85, max_iters=3)
    level, parent = O.bfs(g, 0)
    for mode in ("force_pc", "analytic"):
        r = G.run("pagerank", max_iters=3, mode=mode, profile=True)
        assert r.stats["kernel_launches"][PC_GATHER] == 3
        # a sum of positive FP32 terms in at most three roundings per level, as in the tests of the classes
        assert np.max(np.abs(r.values.cpu().numpy().astype(np.float64) - ref) / ref) <= 1e-5
    for mode in ("force_pc", "force_sc", "analytic"):
        b, d = (G.run(a, source=0, mode=mode, profile=True) for a in ("bfs", "sssp"))
        for r in (b, d):
            launches = r.stats["kernel_launches"]
            assert launches[TASK_GATHER] == r.stats["iterations"]
            assert (launches[PC_GATHER] > 0) == (r.stats["pc_partition_steps"] > 0)
            assert (launches[SC_SCATTER] > 0) == (r.stats["sc_edges_scattered"] > 0)
        assert np.array_equal(b.values.cpu().numpy(), level) and np.array_equal(b.parent.cpu().numpy(), parent)
        assert np.array_equal(d.values.cpu().numpy(), distances(g, 0))
    G.close()


@pytest.mark.parametrize("bits", [8, 24])
def test_split_columns_of_either_weight_format(bits):
    # one column of every edge, split over several tasks whose partial minima are merged
    import paper_1806_08092_gb300 as gp
    n, P, fan = 16384, 1024, 16
    u = np.repeat(np.arange(n, dtype=np.int64), fan)
    v = (u * 37 + np.tile(np.arange(fan, dtype=np.int64), n) * 61) % P
    g = gg.multigraph(n, u.tolist(), v.tolist())
    g.weights = np.random.default_rng(bits).integers(0, 1 << bits, g.num_edges).astype(np.int32)
    g.weights[0] = (1 << bits) - 1
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=P)
    assert G.info()["num_pc_partials"] > 0
    for mode in ("force_pc", "force_sc"):
        r = G.run("sssp", source=5, mode=mode, profile=True)
        assert (r.stats["kernel_launches"][MERGE] > 0) == (mode == "force_pc")
        assert np.array_equal(r.values.cpu().numpy(), distances(g, 5)), mode
    G.close()


def run_counting_frontiers(G, algo, n, source, max_iters, ratio):
    """A run that records its frontiers but not its modes: the iteration's kernels, launched ahead where they may be."""
    from paper_1806_08092_gb300 import _lib
    lib, o, st = _lib.load(), _lib.RunOpts(), _lib.RunStats()
    lib.gpop_run_opts_default(ctypes.byref(o))
    o.algo, o.source, o.max_iters = _lib.ALGOS[algo], source, max_iters
    o.bw_ratio_num, o.bw_ratio_den = ratio, 1
    frontier = np.zeros(2 * max_iters, dtype=np.uint64)
    o.trace_frontier = ctypes.c_void_p(frontier.ctypes.data)
    out = np.zeros(n, dtype=np.uint32)
    _lib.check(lib.gpop_run(G._h, ctypes.byref(o), ctypes.c_void_p(out.ctypes.data), None, 0, ctypes.byref(st)))
    return out, st.as_dict(), frontier.reshape(-1, 2)[:st.iterations]


@pytest.mark.parametrize("ratio", [1, 2, 8])
@pytest.mark.parametrize("algo", ["pagerank", "bfs", "sssp", "cc", "ppr", "nibble"])
def test_launches_ahead_of_the_plan(algo, ratio):
    # iterations of all PC, all SC and mixed partitions follow one another; those launched ahead in vain change nothing
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(14).with_weights()
    if algo == "cc":
        g = gg.symmetrized(g)
    root = int(gg.roots(g, 1)[0])
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights if algo == "sssp" else None, partition_size=512)
    iters = dict(pagerank=12, ppr=25, nibble=25).get(algo, 200)
    kw = dict(source=root, max_iters=iters, bw_ratio=(ratio, 1))
    ahead, stats, frontier = run_counting_frontiers(G, algo, g.num_vertices, root, iters, ratio)
    timed = G.run(algo, trace=True, profile=True, **kw)
    assert np.array_equal(ahead, timed.values.cpu().numpy().view(np.uint32))
    assert np.array_equal(frontier, timed.frontier)
    for key in ("iterations", "converged", "residual", "edges_scattered", "vertices_scattered", "pc_partition_steps",
                "sc_partition_steps", "model_bytes", "sc_vertices_scattered", "sc_edges_scattered", "gathered_vertices"):
        assert stats[key] == timed.stats[key], key
    exact = {"bfs": lambda: O.bfs(g, root)[0], "sssp": lambda: distances(g, root), "cc": lambda: O.cc(g)}
    if algo in exact:
        assert np.array_equal(ahead, exact[algo]())
    G.close()
