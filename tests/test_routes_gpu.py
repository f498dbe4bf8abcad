"""Searches at the sizes where their kernel changes: small graphs in one block,
explicit pushes of graphs that would pull, batches of large directed graphs;
against the CPU oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import test_batch_bc_gpu as tbb
import test_bfs_gpu as tb
from test_small_gpu import star_of_stars

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16383, 16384, 16385])
@pytest.mark.parametrize("direction", ["auto", "push", "pull"])
def test_one_block_up_to_16384_vertices(cuda_lib, n, direction):
    r, c = star_of_stars(n, 1000)
    with cuda_lib.gr_graph_create(r, c) as g:
        for src in (0, 5, n - 1):
            tb.check(cuda_lib, r, c, g, src, tb.opts(cuda_lib, direction))


# 0.43 and 0.78 M entries: below and above what one block takes
@pytest.mark.parametrize("ef", [16, 32])
@pytest.mark.parametrize("direction", ["auto", "push"])
def test_one_block_by_entries(cuda_lib, ef, direction):
    r, c = gg.rmat(14, ef, seed=2)
    assert (c.size <= 1 << 19) == (ef == 16)
    with cuda_lib.gr_graph_create(r, c) as g:
        for src in gg.sources(r, 3, seed=1):
            tb.check(cuda_lib, r, c, g, int(src), tb.opts(cuda_lib, direction))


@pytest.mark.parametrize("keep", [0.7, 0.9])
def test_batch_of_directed_graphs(cuda_lib, keep):
    r, c = gg.rmat(18, 8, seed=3)
    u = np.repeat(np.arange(r.size - 1), np.diff(r))
    arc = np.random.default_rng(1).random(c.size) < keep
    rd = np.zeros_like(r)
    rd[1:] = np.cumsum(np.bincount(u[arc], minlength=r.size - 1))
    cd = c[arc]
    assert (cd.size >= 3_000_000) == (keep == 0.9)
    srcs = gg.sources(rd, 20, seed=2)
    with cuda_lib.gr_graph_create(rd, cd) as g:
        got = tbb.run_batch(cuda_lib, g, srcs)
        for i in range(0, 20, 4):
            assert np.array_equal(got[i], oracle.bfs(rd, cd, int(srcs[i]))[0])
