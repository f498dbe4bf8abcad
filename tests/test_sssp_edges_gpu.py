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
