"""SC messages of the minima and of AND (compacted frontier, equal shares of its edges, one combined word per
destination) at the edges of a share, of the search for its first vertex and of the vertex range, against the oracle.
Kernel timing keeps these small graphs on the iteration's kernels."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    return gp


def check(g, P, root=0, cc=True):
    import paper_1806_08092_gb300 as gp
    g = g.with_weights()
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=P)
    level, parent = O.bfs(g, root)
    dist = O.sssp(g, root)
    d32 = dist.copy()
    d32[dist == O.U64_INF] = O.U32_INF
    src = [root, 1, root, min(7, g.num_vertices - 1)]
    for mode in ("force_sc", "analytic"):
        for rep in range(2):  # the words are at rest again after a run
            r = G.run("bfs", source=root, mode=mode, profile=True)
            assert np.array_equal(r.values.cpu().numpy(), level) and np.array_equal(r.parent.cpu().numpy(), parent), (mode, rep)
            assert np.array_equal(G.run("sssp", source=root, mode=mode, profile=True).values.cpu().numpy(), d32.astype(np.uint32))
            assert np.array_equal(G.run_msbfs(src, mode=mode, profile=True).values.cpu().numpy(), O.msbfs(g, src))
    G.close()
    if cc:
        gs = gg.symmetrized(g)
        H = gp.Graph.from_csr(gs.row_ptr, gs.col, None, partition_size=P)
        for mode in ("force_sc", "analytic"):
            for waves in (0, 3):
                x = H.run("cc", mode=mode, profile=True, isg_waves=waves).values.cpu().numpy()
                assert np.array_equal(x, O.cc(gs)), (mode, waves)
        H.close()


@pytest.mark.parametrize("fan", [1, 1023, 1024, 1025, 2048, 5000])
def test_one_vertex_over_several_shares(fan):
    # vertex 0 reaches fan vertices, which reach one another's successors; the others have no out-edges
    n = 6007
    u = [0] * fan + list(range(1, fan + 1))
    v = list(range(1, fan + 1)) + [(x * 7) % n for x in range(1, fan + 1)]
    check(gg.multigraph(n, u, v), 1024)


@pytest.mark.parametrize("n,P", [(255, 32), (257, 32), (8191, 256), (8193, 256), (70001, 16384), (140003, 4096)])
def test_frontiers_around_the_search_steps(n, P):
    # everyone is active in the first iterations of connected components: lists of n vertices of one to three edges
    rng = np.random.default_rng(n)
    u = np.concatenate([np.arange(n), rng.integers(0, n, n)])
    v = np.concatenate([(np.arange(n) + 1) % n, rng.integers(0, n, n)])
    check(gg.multigraph(n, u.tolist(), v.tolist()), P)
