"""gr_pagerank_stats: what a call that asked for no iteration count did."""
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


def test_iterations_after_the_call(cuda_lib):
    import torch
    gr = cuda_lib
    r, c = gg.rmat(12, 8, seed=3)
    other = torch.cuda.Stream()
    with gr.gr_graph_create(r, c) as g:
        with pytest.raises(gr.GrError) as ei:
            gr.gr_pagerank_stats(g)
        assert ei.value.status == gr.GR_EINVAL
        rank = torch.empty(g.n, dtype=torch.float32, device="cuda")
        for mode in (gr.GR_MODE_AUTO, gr.GR_MODE_LAUNCH):
            for iters in (0, 1, 7):
                assert gr.gr_pagerank(g, rank, 0.85, iters, 0.0, gr.gr_opts(mode=mode),
                                      count=False, stream=other) is None
                assert gr.gr_pagerank_stats(g) == iters
        want = gr.gr_pagerank(g, rank, 0.85, 200, 1e-6)
        assert 1 < want < 200 and gr.gr_pagerank_stats(g) == want
    assert gr._lib.gr_pagerank_stats(None, None) == gr.GR_EINVAL
