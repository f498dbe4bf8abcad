"""Mesh searches run by one block each: the sizes at which their shared-memory
layout changes or no longer fits, hand-over to the grid kernels, statistics
and limits, against the CPU oracle and the other drivers."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import test_bfs_gpu as tb
import test_sssp_gpu as ts

pytestmark = pytest.mark.gpu


def kary_tree(k, n):
    """Vertices in level order, children of v are k v + 1 .. k v + k below n."""
    child = np.arange(1, n)
    parent = (child - 1) // k
    u = np.concatenate([parent, child])
    v = np.concatenate([child, parent])
    at = np.lexsort((v, u))
    r = np.zeros(n + 1, np.int32)
    r[1:] = np.cumsum(np.bincount(u, minlength=n))
    return r, v[at].astype(np.int32)


# the far pile's bits fit beside the near ones up to about 798,000 vertices
@pytest.mark.parametrize("side", [1, 2, 893, 894, 950])
def test_sssp_near_the_far_bits_limit(cuda_lib, side):
    r, c = gg.grid(side, p_del=0.05, seed=side)
    w = gg.weights(r, c, seed=3, wmin=1, wmax=16)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        ts.check(cuda_lib, r, c, w, g, side * side // 3)


# the visited bitmap fits up to 1,589,000 vertices, 1260 x 1260; above, the
# one-cluster driver runs
@pytest.mark.parametrize("side", [1260, 1261, 1300])
def test_bfs_near_the_bitmap_limit(cuda_lib, side):
    r, c = gg.grid(side, p_del=0.05, seed=4)
    with cuda_lib.gr_graph_create(r, c) as g:
        tb.check(cuda_lib, r, c, g, side // 2)


@pytest.mark.parametrize("k,n", [(2, (1 << 21) - 1), (15, 1_700_000)])
def test_bfs_cluster_overflow_and_handoff(cuda_lib, k, n):
    r, c = kary_tree(k, n)
    with cuda_lib.gr_graph_create(r, c) as g:
        for src in (0, n - 1):
            tb.check(cuda_lib, r, c, g, src)


@pytest.mark.parametrize("delta", [0, 16, 0xFFFFFFFF])
def test_sssp_batch_hands_over(cuda_lib, delta):
    """Some lanes outgrow a block, at different thresholds, one does not."""
    r, c = kary_tree(15, 54_241 + 1)  # and a path no tree edge reaches below
    n = r.size - 1
    tail = 300
    r = np.concatenate([r, r[-1] + 2 * np.arange(1, tail + 1)]).astype(np.int32)
    extra = np.stack([np.arange(tail) - 1, np.arange(tail) + 1], 1).clip(0, tail - 1) + n
    c = np.concatenate([c, extra.reshape(-1)]).astype(np.int32)
    w = gg.weights(r, c, seed=21, wmin=1, wmax=64)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        ts.check_batch(cuda_lib, r, c, w, g, [0, n - 1, n + tail // 2, 17, 0],
                       ts.opts(cuda_lib, delta, "persistent"))


def test_sssp_statistics_equal_the_host_driver(cuda_lib):
    n = 513
    r, c = gg.from_edges(n, [(i, i + 1) for i in range(n - 1)])
    w = gg.weights(r, c, seed=2, wmin=1, wmax=9)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        got = []
        for mode in ("persistent", "launch"):
            ts.run_sssp(cuda_lib, g, 3, ts.opts(cuda_lib, 7, mode))
            got.append(cuda_lib.gr_sssp_stats(g))
        assert got[0] == got[1]


def test_limits_are_reported(cuda_lib):
    r, c = gg.grid(60, p_del=0.0)
    w = gg.weights(r, c, seed=2, wmin=1, wmax=9)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        for run, stats in ((ts.run_sssp, cuda_lib.gr_sssp_stats),
                           (tb.run_bfs, cuda_lib.gr_bfs_stats)):
            with pytest.raises(cuda_lib.GrError) as ei:
                run(cuda_lib, g, 0, cuda_lib.gr_opts(mode=cuda_lib.GR_MODE_PERSISTENT, max_iters=5))
                stats(g)
            assert ei.value.status == cuda_lib.GR_ETIMEOUT
        ts.check(cuda_lib, r, c, w, g, 0)  # the graph stays usable
        tb.check(cuda_lib, r, c, g, 0)
