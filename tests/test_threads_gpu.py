"""Calls on graphs of very different size from several host threads, each with a
graph of its own, against the CPU oracle. They share one stream: what meets is
the host side of the calls, not their kernels."""
import threading

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def side_by_side(jobs):
    """Runs the jobs (callables) in a thread each and raises the first error."""
    errors = []
    start = threading.Barrier(len(jobs))

    def body(job):
        try:
            start.wait()
            job()
        except BaseException as e:  # noqa: BLE001 - handed to the caller's thread
            errors.append(e)

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def searches(gr, op, r, c, w, times, s):
    """`times` searches of one kind on one graph on stream s, each compared."""
    import torch
    src = int(gg.sources(r, 1, seed=3)[0])
    want = (oracle.bfs(r, c, src)[0] if op == "bfs"
            else oracle.sssp(r, c, w, src)[0].view(np.int32))

    def job():
        with gr.gr_graph_create(r, c, w) as g, torch.cuda.stream(s):
            out = torch.empty(g.n, dtype=torch.int32, device="cuda")
            for _ in range(times):
                if op == "bfs":
                    gr.gr_bfs(g, src, out, stream=s)
                else:
                    gr.gr_sssp(g, src, out, stream=s)
                s.synchronize()
                assert np.array_equal(out.cpu().numpy(), want)
    return job


# the one-block drivers, whose shared memory follows the graph
@pytest.mark.parametrize("op,kind,small,large", [
    ("bfs", "rmat", 6, 15), ("bfs", "grid", 8, 500), ("sssp", "grid", 8, 500)])
def test_one_block_searches(cuda_lib, op, kind, small, large):
    import torch
    jobs, stream = [], torch.cuda.Stream()
    for size, times in ((small, 400), (large, 100), (small, 400), (large, 100)):
        r, c = gg.rmat(size, 8, seed=3) if kind == "rmat" else gg.grid(size, p_del=0.05, seed=3)
        w = gg.weights(r, c, seed=4, wmin=1, wmax=16) if op == "sssp" else None
        jobs.append(searches(cuda_lib, op, r, c, w, times, stream))
    side_by_side(jobs)
