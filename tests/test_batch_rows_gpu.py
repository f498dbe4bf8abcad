"""Batched BFS pulls over rows of exactly the lengths around an 8-entry group and
a 256-entry tile, against the CPU oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import test_batch_bc_gpu as tb
from test_small_gpu import from_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("row", [1, 7, 8, 9, 255, 256, 257, 511, 512, 513])
@pytest.mark.parametrize("k", [64, 33])
def test_pulled_rows_of_one_length(cuda_lib, row, k):
    # every third vertex of the lower half is joined to `row` of the upper half,
    # the first of which is also joined to all the others there
    n, half = 3000, 1500
    left = np.arange(0, half, 3)
    pairs = [np.stack([np.full(row, v), half + (v * 5 + np.arange(row) * 7) % half], 1)
             for v in left]
    pairs.append(np.stack([np.full(half - 1, half), np.arange(half + 1, n)], 1))
    r, c = from_pairs(n, np.concatenate(pairs))
    deg = np.diff(r)
    assert np.all(deg[left] == row)
    srcs = left[:: left.size // k][:k]
    want = np.stack([oracle.bfs(r, c, int(s))[0] for s in srcs])
    # a level is pulled when its frontier, all lanes together, has a sixteenth of
    # the edges or more: one at least is, with a level after it
    edges = [int(deg[(want == lv).any(0)].sum()) for lv in range(want.max() + 1)]
    assert any(16 * e >= c.size for e in edges[1:-1]), edges
    with cuda_lib.gr_graph_create(r, c) as g:
        assert np.array_equal(tb.run_batch(cuda_lib, g, srcs), want)
