"""What the library does when the runtime refuses it something: a variant of it (faultlib) fails the calls on the host."""
import numpy as np
import pytest

import faultlib
import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def faults(tmp_path_factory):
    import paper_1806_08092_gb300 as gp
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gp.build()
    with faultlib.use(faultlib.build(str(tmp_path_factory.mktemp("faults")))) as f:
        yield f


def check_bfs(G, g, root, **kw):
    r = G.run("bfs", source=root, **kw)
    level, parent = O.bfs(g, root)
    assert np.array_equal(r.values.cpu().numpy(), level) and np.array_equal(r.parent.cpu().numpy(), parent)
    return r


def test_refused_cooperative_launch_takes_the_iterations_kernels(faults):
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(11).with_weights()
    root = int(gg.roots(g, 1)[0])
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=256)
    ref, _, _ = O.pagerank(g, 0.85, max_iters=5)
    for error in (faultlib.COOPERATIVE_LAUNCH_TOO_LARGE, 0, faultlib.COOPERATIVE_LAUNCH_TOO_LARGE):
        with faults.plan(launch_error=error):
            r = check_bfs(G, g, root)
            # one launch visits every vertex in every iteration, the iteration's kernels only columns with messages
            assert (r.stats["gathered_vertices"] < r.stats["iterations"] * g.num_vertices) == (error != 0)
            x = G.run("pagerank", max_iters=5).values.cpu().numpy().astype(np.float64)
            assert np.max(np.abs(x - ref) / ref) <= 1e-5
            src = [root, 1, 2]
            assert np.array_equal(G.run_msbfs(src).values.cpu().numpy(), O.msbfs(g, src))
    G.close()


def allocations(faults, call):
    """How many allocations call() makes."""
    with faults.plan(fail_alloc=1 << 40):
        call()
        return faults.allocs


def test_build_without_memory_for_the_small_graph_layout(faults):
    # every allocation of a build fails once: it reports so, or, where only the layout of the one-launch path is lost, the
    # graph runs by the iteration's kernels
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(9).with_weights()
    root = int(gg.roots(g, 1)[0])

    def build():
        return gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=128)

    whole = build()
    bytes_whole = whole.info()["device_bytes"]
    one = check_bfs(whole, g, root).stats["gathered_vertices"]
    whole.close()
    without = 0
    for n in range(allocations(faults, lambda: build().close())):
        try:
            with faults.plan(fail_alloc=n):
                G = build()
        except gp.GpopError as e:
            assert e.status == 2, n
            continue
        r = check_bfs(G, g, root)
        if r.stats["gathered_vertices"] < one:
            without += 1
            H = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=128)
            check_bfs(H, g, root)
            assert G.info()["device_bytes"] < H.info()["device_bytes"]
            assert np.array_equal(G.run("sssp", source=root).values.cpu().numpy(), H.run("sssp", source=root).values.cpu().numpy())
            H.close()
        G.close()
    assert without >= 9  # its six temporaries, the ranges, the in-edges, their weights
    again = build()
    assert again.info()["device_bytes"] == bytes_whole
    again.close()


def test_call_after_one_without_memory(faults):
    # the failed call's error is its own: the next calls look for theirs and find none
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(9).with_weights()
    root = int(gg.roots(g, 1)[0])
    src = [root, 3]
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=128)
    ways = [lambda: G.run("bfs", source=root, profile=True), lambda: G.run("bfs", source=root, mode="log_both", log_capacity=64),
            lambda: G.run_msbfs(src), lambda: G.run_msbfs(src, device_out=False)]
    G.run("pagerank", max_iters=1, profile=True)
    for way in ways:
        with faults.plan(fail_alloc=0), pytest.raises(gp.GpopError):
            way()
        G.run("pagerank", max_iters=1, profile=True)
        way()
    check_bfs(G, g, root)
    G.close()


def test_in_edges_whose_memory_cannot_be_had(faults):
    # the first batched PPR lays out the in-edges: whichever of its allocations fails, nothing runs on half of them, and
    # the next call starts over
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(9)
    seeds = [int(v) for v in gg.roots(g, 3)]

    def first_call(**plan):
        G = gp.Graph.from_csr(g.row_ptr, g.col, partition_size=128)
        with faults.plan(**plan):
            try:
                return G, G.run_ppr_batch(seeds, max_iters=4).values.cpu().numpy(), faults.allocs
            except gp.GpopError as e:
                assert e.status == 2
                return G, None, faults.allocs

    G, whole, allocs = first_call(fail_alloc=1 << 40)
    G.close()
    for n in range(allocs):
        G, rows, _ = first_call(fail_alloc=n)
        assert rows is None, n
        assert np.array_equal(G.run_ppr_batch(seeds, max_iters=4).values.cpu().numpy(), whole), n
        G.close()


def test_memory_of_failed_allocations_is_not_counted(faults):
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(9).with_weights()
    root = int(gg.roots(g, 1)[0])

    def graph():
        return gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=128)

    def sweep(before, call, falls_back=False):
        """Fails each allocation of call() on a graph prepared by before(): nothing more is counted, or held."""
        G = graph()
        before(G)
        held = G.info()["device_bytes"]
        allocs = allocations(faults, lambda: call(G))
        whole = G.info()["device_bytes"]
        G.close()
        assert allocs > 0 and whole > held
        for n in range(allocs):
            G = graph()
            before(G)
            for _ in range(2):
                with faults.plan(fail_alloc=n):
                    if falls_back:
                        call(G)
                    else:
                        with pytest.raises(gp.GpopError):
                            call(G)
                assert G.info()["device_bytes"] == held, n
            call(G)
            assert G.info()["device_bytes"] == whole, n
            G.close()

    def timed(G):
        check_bfs(G, g, root, profile=True)

    sweep(timed, lambda G: check_bfs(G, g, root), falls_back=True)                # the one-launch path's buffers
    sweep(lambda G: None, lambda G: G.run("pagerank", max_iters=2, profile=True))  # the run's buffers
    sweep(lambda G: G.run("pagerank", max_iters=2, profile=True), timed)           # the SC messages' words


def test_timing_logs_whose_buffers_cannot_be_had(faults):
    # a LOG_BOTH run without memory for its buffers, then one with it
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(9).with_weights()
    root = int(gg.roots(g, 1)[0])
    G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=128)
    check_bfs(G, g, root, profile=True)
    held = G.info()["device_bytes"]
    for n in range(9):
        with faults.plan(fail_alloc=n), pytest.raises(gp.GpopError):
            G.run("bfs", source=root, mode="log_both", log_capacity=64)
        assert G.info()["device_bytes"] == held, n
    r = check_bfs(G, g, root, mode="log_both", log_capacity=64)
    assert r.stats["log_records"] > 0 and G.info()["device_bytes"] > held
    G.close()


def test_build_takes_back_what_its_pool_holds(faults):
    # an allocation that fails while released temporaries lie in the build's pool succeeds once they have gone back
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(9).with_weights()
    root = int(gg.roots(g, 1)[0])

    def build():
        return gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=128)

    for n in range(allocations(faults, lambda: build().close())):
        with faults.plan(fail_alloc=n, until_trim=1):
            G = build()
        check_bfs(G, g, root, profile=True)
        G.close()


def test_first_run_on_a_stream_of_its_own(faults):
    # the run's buffers are cleared on the legacy stream, late here, and the run is on a stream that does not wait for it
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(12).with_weights()
    root = int(gg.roots(g, 1)[0])
    stream = torch.cuda.Stream()
    for mode in ("force_sc", "analytic", "force_pc"):
        G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=256)
        with faults.plan(memset_delay_ms=20), torch.cuda.stream(stream):
            check_bfs(G, g, root, mode=mode, profile=True)
        G.close()


def test_checkpoint_and_run_on_a_stream_of_its_own(faults):
    # the checkpoint's copies are on the legacy stream, late here, and the run that continues it is not
    import paper_1806_08092_gb300 as gp
    g = gg.rmat(12).with_weights()
    root = int(gg.roots(g, 1)[0])
    stream = torch.cuda.Stream()
    want = O.bfs(g, root)[0]
    for profile in (False, True):  # one launch; the iteration's kernels
        G = gp.Graph.from_csr(g.row_ptr, g.col, g.weights, partition_size=256)
        G.run("bfs", source=root, max_iters=2)
        state = G.state_export()
        G.run("bfs", source=(root + 1) % g.num_vertices)
        with faults.plan(copy_delay_ms=20), torch.cuda.stream(stream):
            G.state_import(state)
            r = G.run("bfs", source=root, resume=True, profile=profile)
            assert np.array_equal(r.values.cpu().numpy(), want), profile
        G.close()
