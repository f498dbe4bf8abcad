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
