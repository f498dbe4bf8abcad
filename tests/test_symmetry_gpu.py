"""What a graph handle reports of symmetry when rows repeat a column: every
(u, v) needs a (v, u), however often either is stored."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def csr(n, edges):
    r = np.zeros(n + 1, np.int32)
    np.add.at(r, np.array([u for u, _ in edges], int) + 1, 1)
    return np.cumsum(r).astype(np.int32), np.array([v for _, v in sorted(edges)], np.int32)


CASES = {
    "more_above": (2, [(0, 1), (0, 1), (1, 0)], True),
    "more_below": (3, [(0, 2), (2, 0), (2, 0), (2, 0), (1, 1)], True),
    "balanced": (4, [(0, 1), (0, 1), (1, 0), (2, 3), (3, 2), (3, 2)], True),
    "one_way_among_repeats": (4, [(0, 1), (0, 1), (1, 0), (2, 3), (3, 1)], False),
    "one_way_balanced": (4, [(0, 1), (0, 1), (1, 0), (3, 2)], False),
    "repeated_self_loop": (2, [(0, 0), (0, 0), (0, 1), (1, 0)], True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_repeated_entries(cuda_lib, name):
    import torch
    gr = cuda_lib
    n, edges, want = CASES[name]
    r, c = csr(n, edges)
    with gr.gr_graph_create(r, c) as g:
        assert gr.gr_graph_info(g)["symmetric"] == want
        # a pull, PPR and CC go by it
        d = torch.empty(n, dtype=torch.int32, device="cuda")
        if want:
            gr.gr_bfs(g, 0, d, None, gr.gr_opts(direction=gr.GR_DIR_PULL))
            assert np.array_equal(d.cpu().numpy(), oracle.bfs(r, c, 0)[0])
            gr.gr_ppr(g, [0], torch.empty(n, dtype=torch.float64, device="cuda"), max_iter=2)
        else:
            with pytest.raises(gr.GrError) as ei:
                gr.gr_bfs(g, 0, d, None, gr.gr_opts(direction=gr.GR_DIR_PULL))
            assert ei.value.status == gr.GR_EINVAL
        gr.gr_cc(g, d)
        assert np.array_equal(d.cpu().numpy(), oracle.cc(r, c)[0])


def test_bipartite_with_repeats(cuda_lib):
    import torch
    r, c = csr(3, [(0, 2), (0, 2), (1, 2), (2, 0), (2, 1)])
    with cuda_lib.gr_graph_create(r, c) as g:
        score = torch.empty(3, dtype=torch.float64, device="cuda")
        assert cuda_lib.gr_hits(g, 2, score, max_iter=3, tol=0.0) == 3
