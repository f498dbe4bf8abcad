"""The batched kernels where a lane word, a warp's group or a tile ends: lane
counts around half a word, levels of one vertex and of a few more than the
finish takes per warp, rows around the 256-entry pull tiles, against the CPU
oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import test_batch_bc_gpu as tb
from test_small_gpu import from_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 31, 32, 33, 63, 64])
def test_lane_counts(cuda_lib, k):
    r, c = gg.rmat(11, 8, seed=k)
    srcs = gg.sources(r, k, seed=k)
    with cuda_lib.gr_graph_create(r, c) as g:
        d = tb.run_batch(cuda_lib, g, srcs)
        for i in range(k):
            assert np.array_equal(d[i], oracle.bfs(r, c, int(srcs[i]))[0]), f"lane {i}"
        tb.check_bc(tb.run_bc(cuda_lib, g, srcs), oracle.bc(r, c, srcs))


@pytest.mark.parametrize("per_warp,extra", [(0, 1), (1, -1), (1, 1), (3, 5), (5, 0), (8, 3)])
def test_bc_levels_of_every_group_size(cuda_lib, per_warp, extra):
    import torch
    warps = 64 * torch.cuda.get_device_properties(0).multi_processor_count
    q = per_warp * warps + extra  # vertices of the level that has children
    mid = np.arange(2, 2 + q)
    pairs = np.concatenate([[[0, 1]], np.stack([np.full(q, 1), mid], 1),
                            np.stack([mid, mid + q], 1),
                            np.stack([mid[:-1], mid[1:] + q], 1)])
    r, c = from_pairs(2 + 2 * q, pairs)
    srcs = [0, 1, 0]
    with cuda_lib.gr_graph_create(r, c) as g:
        tb.check_bc(tb.run_bc(cuda_lib, g, srcs), oracle.bc(r, c, srcs))


@pytest.mark.parametrize("row", [1, 7, 8, 9, 255, 256, 257, 513])
def test_batched_pull_of_rows_around_a_tile(cuda_lib, row):
    # rows of `row` entries in a graph dense enough to be pulled, one of many
    # tiles, and vertices without edges between them
    rng = np.random.default_rng(row)
    n = 3000
    left = np.repeat(np.arange(0, n // 2, 3), row)
    pairs = np.concatenate([np.stack([left, rng.integers(n // 2, n, left.size)], 1),
                            np.stack([np.full(n // 2, n // 2), np.arange(n // 2, n)], 1)])
    r, c = from_pairs(n, pairs)
    srcs = gg.sources(r, 64, seed=row)
    with cuda_lib.gr_graph_create(r, c) as g:
        d = tb.run_batch(cuda_lib, g, srcs)
        for i in range(64):
            assert np.array_equal(d[i], oracle.bfs(r, c, int(srcs[i]))[0]), f"lane {i}"
