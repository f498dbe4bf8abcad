"""What SSSP starts out with on a graph, by its degrees and size."""
import numpy as np
import pytest

import graphgen as gg
from test_sssp_edges_gpu import regular

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,means,blocks", [
    (lambda: gg.grid(60, p_del=0.05, seed=1), 6, 1),
    (lambda: regular(2000, 8, 1), 6, 1),        # degree 16
    (lambda: regular(2000, 10, 1), 2, 1),       # 20, too few entries to pull
    (lambda: regular(100_000, 10, 1), 2, 2),    # pulled: two blocks per SM
    (lambda: gg.rmat(12, 16, seed=1), 8, 1)])
def test_bucket_and_grid(cuda_lib, make, means, blocks):
    gr = cuda_lib
    r, c = make()
    w = gg.weights(r, c, seed=3, wmin=1, wmax=64)
    with gr.gr_graph_create(r, c, w) as g:
        t = gr.gr_tuned_sssp(g)
    mean = int(w.sum(dtype=np.uint64)) / w.size
    assert t["mode"] == gr.GR_MODE_PERSISTENT
    assert t["delta"] == int(means * mean) and t["blocks_per_sm"] == blocks
