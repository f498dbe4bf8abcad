"""SSSP where a workspace, a limit or a layout changes under the search, against
the CPU oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import test_sssp_gpu as ts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def s12w(cuda_lib):
    r, c = gg.rmat(12, 16, seed=6)
    w = gg.weights(r, c, seed=7, wmin=1, wmax=64)
    g = cuda_lib.gr_graph_create(r, c, w)
    yield r, c, w, g
    g.close()


@pytest.mark.parametrize("mode", ["persistent", "launch", "graph"])
@pytest.mark.parametrize("direction,alpha", [("auto", 16.0), ("pull", 0.0)])
def test_one_source_after_a_larger_batch(cuda_lib, s12w, mode, direction, alpha):
    """A workspace of many lanes cannot pull, one of one lane can."""
    r, c, w, _ = s12w
    srcs = [int(x) for x in gg.sources(r, 16, seed=8)]
    o = ts.opts(cuda_lib, 0, mode, direction, alpha)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        for k in (1, 16, 1, 2, 1):
            ts.check_batch(cuda_lib, r, c, w, g, srcs[:k], o)


@pytest.mark.parametrize("mode", ["launch", "persistent", "graph"])
@pytest.mark.parametrize("direction", ["pull", "push", "auto"])
def test_every_iteration_limit(cuda_lib, mode, direction):
    """A search either ends within its limit, with the right distances, or
    reports that it did not, whatever the launches an iteration takes."""
    # a path through hubs of 20 leaves each: 40 relaxations, one bucket
    hubs = 40
    edges = [(i, i + 1) for i in range(hubs - 1)]
    edges += [(i, hubs + 20 * i + j) for i in range(hubs) for j in range(20)]
    r, c = gg.from_edges(hubs * 21, edges)
    w = gg.weights(r, c, seed=3, wmin=1, wmax=64)
    want = oracle.sssp(r, c, w, 0)[0]
    o = ts.opts(cuda_lib, 0xFFFFFFFF, mode, direction, 100.0 if direction == "auto" else 0.0)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        for limit in list(range(1, 12)) + [20, 21, 22, 23, 30, 38, 39, 40, 41, 42, 100]:
            o.max_iters = limit
            try:
                d, _ = ts.run_sssp(cuda_lib, g, 0, o, with_pred=False)
            except cuda_lib.GrError as e:
                assert e.status == cuda_lib.GR_ETIMEOUT and limit < 42, limit
                continue
            assert np.array_equal(d, want), limit
            # a push goes one step further an iteration, and finds its end in
            # one more; a pull may go further
            assert direction != "push" or limit >= hubs, limit


def regular(n, half, seed):
    """`half` random permutations and their inverses: degrees up to 2 * half."""
    rng = np.random.default_rng(seed)
    u, v = np.tile(np.arange(n), half), np.concatenate([rng.permutation(n) for _ in range(half)])
    key = np.unique(np.concatenate([u * n + v, v * n + u]))
    key = key[key // n != key % n]
    r = np.zeros(n + 1, np.int32)
    r[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    return r, (key % n).astype(np.int32)


# frontiers that outgrow a block at once; the far pile's bits in shared memory or
# not, rows of four and of more entries
@pytest.mark.parametrize("n,half", [(30_000, 2), (30_000, 3), (30_000, 8), (900_000, 2),
                                    (900_000, 4)])
def test_hand_over_of_random_graphs(cuda_lib, n, half):
    r, c = regular(n, half, half)
    w = gg.weights(r, c, seed=3, wmin=0, wmax=64)
    srcs = [int(x) for x in gg.sources(r, 3, seed=4)]
    with cuda_lib.gr_graph_create(r, c, w) as g:
        for delta in (0, 1, 200, 0xFFFFFFFF):
            o = ts.opts(cuda_lib, delta, "persistent")
            ts.check(cuda_lib, r, c, w, g, srcs[0], o)
        ts.check_batch(cuda_lib, r, c, w, g, srcs)


def test_wide_buckets_are_for_thin_frontiers(cuda_lib):
    """A search of a random graph of degree 16 expands about as many edges in the
    graph's own bucket widths as in two mean weights; a mesh takes fewer
    iterations."""
    r, c = regular(100_000, 8, 1)
    w = gg.weights(r, c, seed=3, wmin=1, wmax=64)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        ts.run_sssp(cuda_lib, g, 5, with_pred=False)
        own = cuda_lib.gr_sssp_stats(g)[2]
        ts.run_sssp(cuda_lib, g, 5, ts.opts(cuda_lib, 65, "persistent"), with_pred=False)
        assert own < 1.25 * cuda_lib.gr_sssp_stats(g)[2]
    r, c = gg.grid(200, p_del=0.05, seed=4)
    w = gg.weights(r, c, seed=3, wmin=1, wmax=64)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        ts.run_sssp(cuda_lib, g, 5, with_pred=False)
        own = cuda_lib.gr_sssp_stats(g)[0]
        ts.run_sssp(cuda_lib, g, 5, ts.opts(cuda_lib, 65, "persistent"), with_pred=False)
        assert own < 0.95 * cuda_lib.gr_sssp_stats(g)[0]
