"""Forced SC and PC modes run the scatters they name on every graph, small ones too: the counts and bits of a plain run are
those of a run whose kernels are timed, which lists the launches, and the results are the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COUNTS = ["iterations", "converged", "edges_scattered", "vertices_scattered", "pc_partition_steps", "sc_partition_steps",
          "model_bytes", "sc_vertices_scattered", "sc_edges_scattered", "gathered_vertices"]
SC_SCATTER, PC_GATHER = 2, 4  # kinds of kernel_launches


@pytest.fixture(scope="module", autouse=True)
def lib():
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    return gp


@pytest.mark.parametrize("P", [32, 512])
@pytest.mark.parametrize("mode", ["force_sc", "force_pc"])
def test_forced_modes_run_their_scatters_on_small_graphs(mode, P):
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(12).with_weights()
    root = int(gg.roots(g, 1)[0])
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=P)
    dist = O.sssp(g, root)
    dist = np.where(dist == O.U64_INF, O.U32_INF, dist).astype(np.uint32)
    exact = {"bfs": O.bfs(g, root)[0], "sssp": dist}
    for algo, kw in (("pagerank", dict(max_iters=6)), ("pagerank", dict(max_iters=6, msg_bf16=True)), ("bfs", dict(source=root)),
                     ("sssp", dict(source=root)), ("ppr", dict(source=root, max_iters=8)),
                     ("nibble", dict(source=root, epsilon=1e-4, max_iters=20))):
        G.run(algo, mode=mode, **kw)  # which data rows a run must clear depends on the run before it
        plain, timed = G.run(algo, mode=mode, **kw), G.run(algo, mode=mode, profile=True, **kw)
        launches = timed.stats["kernel_launches"]
        assert (launches[SC_SCATTER] > 0) == (mode == "force_sc") and (launches[PC_GATHER] > 0) == (mode == "force_pc"), algo
        for key in COUNTS:
            assert plain.stats[key] == timed.stats[key], (algo, key)
        assert np.array_equal(plain.values.cpu().numpy().view(np.uint32), timed.values.cpu().numpy().view(np.uint32)), algo
        if algo in exact:
            assert np.array_equal(plain.values.cpu().numpy(), exact[algo]), algo
    src = [int(v) for v in gg.roots(g, 5)]
    a, b = G.run_msbfs(src, mode=mode), G.run_msbfs(src, mode=mode, profile=True)
    assert np.array_equal(a.values.cpu().numpy(), O.msbfs(g, src))
    assert a.stats["gathered_vertices"] == b.stats["gathered_vertices"]
    G.close()
