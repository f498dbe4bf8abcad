"""How many SSSP requests of one graph the server runs as one search: its lane
limit follows from what a lane adds, not from what a graph holds once."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def test_large_mesh_takes_64_lanes(cuda_lib):
    import torch
    gr = cuda_lib
    side = 1260  # 64 lanes of 36 bytes a vertex: 3.7 of the 4 GB
    r, c = gg.grid(side, p_del=0.05, seed=4)
    w = gg.weights(r, c, seed=5, wmin=1, wmax=16)
    srcs = [int(x) for x in gg.sources(r, 65, seed=6)]
    with gr.gr_graph_create(r, c, w) as g, gr.gr_server_create(16 << 30, 1, 64) as srv:
        gid = gr.gr_server_add_graph(srv, g, True)
        outs = [torch.empty(g.n, dtype=torch.int32, device="cuda") for _ in srcs]
        # the first runs alone, a few ms and the making of its workspace; the
        # others queue meanwhile
        for s, o in zip(srcs, outs):
            gr.gr_server_submit(srv, gid, gr.GR_QUERY_SSSP, s, o)
        gr.gr_server_drain(srv, 120000)
        st = gr.gr_server_stats(srv)
        assert st["completed"] == 65 and st["failed"] == 0 and st["launches"] == 2
        for s, o in list(zip(srcs, outs))[::32]:
            assert np.array_equal(o.cpu().numpy().view(np.uint32), oracle.sssp(r, c, w, s)[0])
