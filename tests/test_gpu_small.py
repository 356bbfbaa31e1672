"""Small graphs run in one launch; the same calls with kernel timing run the iteration's kernels.  Both must agree:
values (exactly, or to FP32 rounding for the sums), iterations and every count of the statistics."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COUNTS = ["iterations", "converged", "edges_scattered", "vertices_scattered", "pc_partition_steps", "sc_partition_steps",
          "model_bytes", "sc_vertices_scattered", "sc_edges_scattered"]


@pytest.fixture(scope="module", autouse=True)
def lib():
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    return gp


def hubs(n, fan, seed=1):
    """A few destinations whose in-edges span several warps' shares, among many of one or two."""
    rng = np.random.default_rng(seed)
    u = np.concatenate([rng.integers(0, n, fan), rng.integers(0, n, fan // 3), rng.integers(0, n, 4 * n)])
    v = np.concatenate([np.full(fan, 5), np.full(fan // 3, n - 1), rng.integers(0, n, 4 * n)])
    return gg.multigraph(n, u.tolist(), v.tolist())


GRAPHS = [("one", gg.multigraph(1, [0], [0]), 32), ("ring", gg.ring(100), 32), ("star", gg.star(3000), 256),
          ("ragged", gg.uniform(3001, 20000), 64), ("sinks", gg.uniform(2500, 3000), 1024), ("hubs", hubs(20011, 7000), 2048),
          ("rmat14", gg.rmat(14), 1024), ("rmat17", gg.rmat(17), 16384), ("sparse", gg.uniform(500009, 600000), 16384)]


@pytest.mark.parametrize("name,g,P", GRAPHS, ids=[x[0] for x in GRAPHS])
def test_one_launch_agrees_with_iteration_kernels(name, g, P):
    import paper_1806_08092_gb300 as gp
    g = g.with_weights()
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=P)
    root = int(gg.roots(g, 1)[0])
    runs = [("pagerank", dict(max_iters=12)), ("pagerank", dict(max_iters=12, msg_bf16=True)), ("bfs", dict(source=root)),
            ("cc", {}), ("sssp", dict(source=root)), ("ppr", dict(source=root, max_iters=15)),
            ("nibble", dict(source=root, epsilon=0.0, max_iters=6))]
    for algo, kw in runs:
        for mode in ("analytic", "force_sc", "force_pc"):
            a, b = G.run(algo, mode=mode, **kw), G.run(algo, mode=mode, profile=True, **kw)
            x, y = a.values.cpu().numpy(), b.values.cpu().numpy()
            if algo in ("pagerank", "ppr", "nibble"):
                # FP32 sums of at most 7000 positive messages in two orders, compounded over the iterations; BF16
                # messages may round the other way where their values differ by a rounding
                tol = 2.0 ** -7 if kw.get("msg_bf16") else 1e-5
                big = y > 1e-12
                assert np.max(np.abs(x.astype(np.float64) - y)[big] / y[big], initial=0) <= tol, (algo, mode)
                assert np.max(np.abs(x.astype(np.float64) - y)[~big], initial=0) <= 1e-12
            else:
                assert np.array_equal(x, y), (algo, mode)
                if algo == "bfs":
                    assert np.array_equal(a.parent.cpu().numpy(), b.parent.cpu().numpy())
            for key in COUNTS:
                assert a.stats[key] == b.stats[key], (algo, mode, key)
    src = [root] * 2 + [int(v) for v in gg.roots(g, 35)]
    lv = G.run_msbfs(src).values.cpu().numpy()
    assert np.array_equal(lv, G.run_msbfs(src, profile=True).values.cpu().numpy())
    if g.num_vertices < 50000:
        assert np.array_equal(lv, O.msbfs(g, src))
    G.close()


@pytest.mark.parametrize("algo", ["pagerank", "bfs", "sssp", "ppr"])
def test_split_runs_cross_both_paths(algo):
    # iterations 1-2 in one launch, 3-4 by the iteration's kernels, the rest in one launch again
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(13).with_weights()
    root = int(gg.roots(g, 1)[0])
    kw = {} if algo == "pagerank" else dict(source=root)
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=512)
    whole = G.run(algo, max_iters=9, **kw)
    G.run(algo, max_iters=2, **kw)
    G.run(algo, max_iters=2, resume=True, profile=True, **kw)
    state = G.state_export()
    H = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=512)
    H.state_import(state)
    last = H.run(algo, max_iters=5, resume=True, **kw)
    x, y = last.values.cpu().numpy(), whole.values.cpu().numpy()
    if algo in ("pagerank", "ppr"):
        assert np.max(np.abs(x.astype(np.float64) - y)) <= 1e-6 * float(np.max(y))  # FP32 sums in two orders
    else:
        assert np.array_equal(x, y)
    host = G.run(algo, max_iters=9, device_out=False, **kw)
    assert np.array_equal(host.values, y)
    G.close()
    H.close()
