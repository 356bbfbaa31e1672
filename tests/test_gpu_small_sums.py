"""Sums of the one-launch path at a hub of nearly the largest in-degree it takes, and where few bits decide.

Every vertex's messages are added without loss beyond their own rounding and rounded to FP32 once: the sum (a pair of FP32
words per destination) differs from the exact one by at most n 2^-48 of it for n positive messages, so its FP32 value is
the exact sum's, or, where that lies within n 2^-48 of the middle of two FP32 numbers (n 2^-23 of all cases: 0.4 % for the
hub of 30000, one in 100000 for the others), its neighbour."""
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


def hub_graph(n, fan, others, seed):
    rng = np.random.default_rng(seed)
    u = np.concatenate([rng.choice(n, fan, replace=False), rng.integers(0, n, others)])
    v = np.concatenate([np.full(fan, 7), rng.integers(0, n, others)])
    u[:fan // 4] = u[0]  # repeated edges: one source's message many times
    return gg.multigraph(n, u.tolist(), v.tolist())


@pytest.mark.parametrize("n,fan,others", [(40009, 30000, 1900000), (5000, 2000, 30000), (300, 4, 20000)])
def test_sums_are_rounded_once(n, fan, others):
    import paper_1806_08092_gb300 as gp
    g = hub_graph(n, fan, others, n)
    G = gp.Graph.from_csr(g.row_ptr, g.col, partition_size=1024)
    r = G.run("pagerank", max_iters=1)
    assert sum(r.stats["kernel_launches"]) == 0 and r.stats["gathered_vertices"] == n  # one launch for the run
    x = r.values.cpu().numpy()
    deg = np.diff(g.row_ptr.astype(np.int64))
    src = np.repeat(np.arange(n), deg)
    first = np.float32(1.0) / np.float32(n)
    msg = np.where(deg > 0, first / np.maximum(deg, 1).astype(np.float32), np.float32(0.0)).astype(np.float32)
    total = np.zeros(n)
    np.add.at(total, g.col.astype(np.int64), msg[src].astype(np.float64))
    c0, c1 = np.float32((1.0 - 0.85) / n), np.float32(0.85)

    def value(s):  # one fused multiply-add: the product of two FP32 numbers is exact in FP64
        return (np.float64(c1) * s.astype(np.float64) + np.float64(c0)).astype(np.float32)

    rounded = total.astype(np.float32)
    assert np.count_nonzero(x != value(rounded)) <= 4
    lo, hi = value(np.nextafter(rounded, np.float32(0))), value(np.nextafter(rounded, np.float32(1)))
    assert np.all((lo <= x) & (x <= hi))
    G.close()


def test_nibble_threshold_decides_alike_on_both_paths():
    # messages of at least epsilon / 2 are exact in the SC scatter's fixed point as in the one-launch path's pairs: values
    # agree to FP32 rounding compounded over the iterations, and the frontiers are the same
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(13)
    G = gp.Graph.from_csr(g.row_ptr, g.col, partition_size=512)
    for root in gg.roots(g, 4):
        for eps in (1e-4, 1e-6):
            kw = dict(source=int(root), epsilon=eps, max_iters=60)
            a, b = G.run("nibble", **kw), G.run("nibble", mode="force_sc", profile=True, **kw)
            for key in ("iterations", "converged", "vertices_scattered", "edges_scattered"):
                assert a.stats[key] == b.stats[key], (root, eps, key)
            x, y = a.values.cpu().numpy().astype(np.float64), b.values.cpu().numpy().astype(np.float64)
            assert np.max(np.abs(x - y)) <= 60 * 2.0 ** -23 * np.max(y)
            ref, _, _ = O.nibble(g, int(root), eps, max_iters=60)
            assert np.max(np.abs(x - ref)) <= 1e-5 * np.max(ref)
    G.close()
