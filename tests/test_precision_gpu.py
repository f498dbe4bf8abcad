"""Results that rest on FP64 arithmetic, bit for bit against numpy's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# a hub with arcs to k of n vertices; chosen so that damping * sum + base lies so
# near the middle of two floats that 48 bits of it round the other way
@pytest.mark.parametrize("n,damping,k", [
    (724, 0.8862, 66), (1374, 0.8201, 9), (1036, 0.7808, 786), (4291, 0.8408, 27),
    (5024, 0.7253, 229), (7182, 0.9853, 99), (4939, 0.1109, 387), (5785, 0.2359, 149)])
def test_pagerank_rounds_the_fp64_rank(cuda_lib, n, damping, k):
    import torch
    r = np.full(n + 1, k, np.int32)
    r[0] = 0
    c = np.arange(1, k + 1, dtype=np.int32)
    rank = torch.empty(n, dtype=torch.float32, device="cuda")
    with cuda_lib.gr_graph_create(r, c) as g:
        cuda_lib.gr_pagerank(g, rank, damping, 1, 0.0)
    got = rank.cpu().numpy()
    d = np.float64(np.float32(damping))
    base = (1.0 - d) / n + d * ((n - 1.0) / n) / n  # all but the hub are dangling
    share = np.float64((np.float32(1) / np.float32(n)) / np.float32(k))
    assert np.all(got[1:k + 1] == np.float32(base + d * share))
    assert got[0] == np.float32(base) and np.all(got[k + 1:] == np.float32(base))


@pytest.mark.parametrize("hubs", [1, 3, 1000])
def test_ppr_divides_by_the_degree(cuda_lib, hubs):
    """One iteration from `hubs` seeds of degrees 1, 2, ... (a star each): a leaf
    of degree one gets damping times what its hub's rank over its degree is, which
    the kernel forms from the degree's reciprocal."""
    import torch
    gr = cuda_lib
    deg = np.arange(1, hubs + 1)
    leaves = int(deg.sum())
    n = hubs + leaves
    hub_of = np.repeat(np.arange(hubs), deg)
    r = np.zeros(n + 1, np.int32)
    r[1:hubs + 1] = np.cumsum(deg)
    r[hubs + 1:] = leaves + np.arange(1, leaves + 1)
    c = np.concatenate([np.arange(hubs, n), hub_of]).astype(np.int32)
    rank = torch.empty(n, dtype=torch.float64, device="cuda")
    for damping in (0.85, 0.3):
        with gr.gr_graph_create(r, c) as g:
            gr.gr_ppr(g, list(range(hubs)), rank, damping, 1, 0.0)
        want = damping * ((1.0 / hubs) / deg)[hub_of]
        assert np.array_equal(rank.cpu().numpy()[hubs:], want)
