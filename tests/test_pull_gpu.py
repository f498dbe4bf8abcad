"""Pull levels of the grid's BFS at the edges of a warp's share: one visited
word per warp and one more, the 32 words of a step and one more, a ragged last
word, long lists, and the pushes that follow a pull, against the CPU oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import test_bfs_gpu as tb
from test_small_gpu import from_pairs

pytestmark = pytest.mark.gpu


def skewed(n, seed):
    """Random pairs, one end skewed to low ids, then renumbered: rows of one to
    thousands of entries, and vertices without any."""
    rng = np.random.default_rng(seed)
    k = 3 * n
    u = (n * rng.random(k) ** 4).astype(np.int64)
    ids = rng.permutation(n)
    return from_pairs(n, ids[np.stack([u, rng.integers(0, n, k)], 1)])


@pytest.mark.parametrize("words,extra", [(1, -31), (1, 0), (1, 1), (3, 5), (32, 0), (32, 33)])
def test_pull_at_the_edges_of_a_warps_words(cuda_lib, words, extra):
    import torch
    warps = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    n = words * 32 * warps + extra  # words per warp at one block per SM
    r, c = skewed(n, words + 100)
    src = int(gg.sources(r, 1, seed=3)[0])
    with cuda_lib.gr_graph_create(r, c) as g:
        for direction, mode, block in [("auto", "persistent", 1), ("pull", "persistent", 1),
                                       ("auto", "persistent", 4), ("auto", "graph", 0),
                                       ("pull", "launch", 0)]:
            tb.check(cuda_lib, r, c, g, src, tb.opts(cuda_lib, direction, mode, block=block))
            assert cuda_lib.gr_bfs_stats(g)[1] > 0
        # pull only while the frontier is nearly everything: pushes follow it
        # from small and from large segments
        for beta in (1.01, 1e9):
            tb.check(cuda_lib, r, c, g, src,
                     tb.opts(cuda_lib, "auto", "persistent", block=2, alpha=1e6, beta=beta))


def test_a_hub_found_by_a_pull_is_pushed_from_the_queue(cuda_lib):
    # the source's 40 neighbours are pulled from; they find a hub of 5000
    # leaves and little else, so that the next level pushes the hub
    n = 60_000
    hub, leaves = 50_000, np.arange(50_001, 55_001)
    near = np.arange(1, 41)
    far = np.arange(55_001, n - 1)
    r, c = from_pairs(n, np.concatenate([
        np.stack([np.zeros(40, int), near], 1), np.stack([near, np.full(40, hub)], 1),
        np.stack([np.full(5000, hub), leaves], 1), np.stack([far[:-1], far[1:]], 1)[::2]]))
    with cuda_lib.gr_graph_create(r, c) as g:
        for block in (1, 4):
            o = tb.opts(cuda_lib, "auto", "persistent", block=block, alpha=1e6, beta=1.01)
            tb.check(cuda_lib, r, c, g, 0, o)
