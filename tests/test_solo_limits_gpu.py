"""The largest meshes that the one-block drivers take and the first they do not:
32 vertices to a bitmap word, 58112 words of shared memory less 16 for the
kernels' own state."""
import numpy as np
import pytest

import graphgen as gg
import test_bfs_gpu as tb
import test_sssp_gpu as ts

pytestmark = pytest.mark.gpu

QUEUES = 2 * 4096  # words
WORDS = 58112 - 16 - QUEUES
SSSP_BOTH = WORDS // 2 * 32  # near and far bits
SSSP_NEAR = WORDS * 32       # near bits alone
BFS = (WORDS - 32) * 32      # visited bits and a spare word a lane


def strip(n, width=1000):
    """A grid of `width` columns cut off after n vertices."""
    v = np.arange(n)
    right, down = v[:-1][(v[:-1] + 1) % width != 0], v[:n - width]
    u = np.concatenate([right, right + 1, down, down + width])
    x = np.concatenate([right + 1, right, down + width, down])
    at = np.argsort(u * n + x)
    r = np.zeros(n + 1, np.int32)
    r[1:] = np.cumsum(np.bincount(u, minlength=n))
    return r, x[at].astype(np.int32)


# beyond the limits up to what the shared memory would hold without the state
@pytest.mark.parametrize("n", [lim + d for lim in (SSSP_BOTH, SSSP_NEAR)
                               for d in (0, 1, 96, 160, 192, 193, 512)])
def test_sssp_sizes(cuda_lib, n):
    r, c = strip(n)
    w = gg.weights(r, c, seed=3, wmin=1, wmax=16)
    with cuda_lib.gr_graph_create(r, c, w) as g:
        ts.check(cuda_lib, r, c, w, g, n // 3)


@pytest.mark.parametrize("n", [BFS - 31, BFS, BFS + 1, BFS + 512, 1263 ** 2, 1264 ** 2])
def test_bfs_sizes(cuda_lib, n):
    r, c = strip(n)
    with cuda_lib.gr_graph_create(r, c) as g:
        tb.check(cuda_lib, r, c, g, n // 3)


def grid3(s):
    at = np.arange(s ** 3).reshape(s, s, s)
    u = np.concatenate([at[:-1].ravel(), at[:, :-1].ravel(), at[:, :, :-1].ravel()])
    v = np.concatenate([at[1:].ravel(), at[:, 1:].ravel(), at[:, :, 1:].ravel()])
    key = np.sort(np.concatenate([u * s ** 3 + v, v * s ** 3 + u]))
    r = np.zeros(s ** 3 + 1, np.int32)
    r[1:] = np.cumsum(np.bincount(key // s ** 3, minlength=s ** 3))
    return r, (key % s ** 3).astype(np.int32)


# rows of six entries: 500,000 entries in all are where the cluster takes over
@pytest.mark.parametrize("side", [43, 44, 45])
def test_bfs_of_3d_grids(cuda_lib, side):
    r, c = grid3(side)
    assert (c.size * 6 <= 3_000_000) == (side < 45)
    with cuda_lib.gr_graph_create(r, c) as g:
        for src in (0, side ** 3 // 2):
            tb.check(cuda_lib, r, c, g, src)
