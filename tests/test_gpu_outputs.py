"""Result buffers that are no whole words of the GPU's memory, which a copy takes, on small and on other paths."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("profile", [False, True])  # one launch for the run; the iteration's kernels
def test_results_at_any_address(offset, profile):
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    g = gg.rmat(10)
    n = g.num_vertices
    root = int(gg.roots(g, 1)[0])
    G = gp.Graph.from_csr(g.row_ptr, g.col, partition_size=64)
    level, parent = O.bfs(g, root)
    whole = G.run("pagerank", max_iters=4, profile=profile).values.cpu().numpy()

    def buffer():
        raw = torch.full((4 * n + 16,), 0xAB, dtype=torch.uint8, device="cuda")
        return raw, raw[offset:offset + 4 * n]

    def check(raw, want):
        b = raw.cpu().numpy()
        assert np.array_equal(b[offset:offset + 4 * n], np.ascontiguousarray(want).view(np.uint8))
        assert np.all(b[:offset] == 0xAB) and np.all(b[offset + 4 * n:] == 0xAB)

    (r0, out), (r1, par) = buffer(), buffer()
    G.run("bfs", source=root, out=out, out_parent=par, profile=profile)
    check(r0, level)
    check(r1, parent)
    r2, out = buffer()
    G.run("pagerank", max_iters=4, out=out, profile=profile)
    check(r2, whole)
    G.close()
