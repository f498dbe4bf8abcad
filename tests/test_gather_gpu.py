"""The all-vertex gather-reduce at the edges of its tiles: rows of every
length around the 8-entry groups, the 256- and 512-entry tiles and their
multiples, with empty rows between them, against the CPU oracle."""
import numpy as np
import pytest

import oracle
from checks import relative_l1
from test_rank_gpu import sum_bound

pytestmark = pytest.mark.gpu

# row lengths in order; 0 is a vertex without entries
ROWS = {
    "one_entry": [1],
    "one_group": [0, 8, 0],
    "groups": [7, 1, 8, 9, 0, 15, 16, 17],
    "tile_less_one": [255],
    "tile": [256, 0, 256],
    "tile_plus_one": [257, 255, 0, 1, 511, 512, 513],
    "over_many_tiles": [3, 5000, 0, 0, 2, 4097, 1],
    "short_rows": [1 + (i * 7) % 5 if i % 3 else 0 for i in range(3000)],
    "mixed": [(i * i * 31) % 97 for i in range(400)] + [2048, 0, 1024, 1],
}


def csr(lengths, n):
    """A directed CSR with rows of the given lengths over n >= len vertices."""
    lengths = np.array(lengths + [0] * (n - len(lengths)), dtype=np.int64)
    r = np.zeros(n + 1, np.int32)
    r[1:] = np.cumsum(lengths)
    c = np.concatenate([np.sort((np.arange(k) * 13 + v * 5) % n) for v, k in enumerate(lengths)])
    return r, c.astype(np.int32)


@pytest.mark.parametrize("name", list(ROWS))
def test_rows_at_tile_edges(cuda_lib, name):
    import torch
    gr = cuda_lib
    n = max(len(ROWS[name]), 7)
    r, c = csr(ROWS[name], n)
    rng = np.random.default_rng(len(c))
    w = rng.integers(0, 2**32, c.size, dtype=np.uint32)
    xf = rng.standard_normal(n)
    xi = rng.integers(-2**31, 2**31, n).astype(np.int32)
    with gr.gr_graph_create(r, c, w) as g:
        for op in (gr.GR_REDUCE_SUM, gr.GR_REDUCE_WSUM, gr.GR_REDUCE_MIN, gr.GR_REDUCE_MAX):
            is_sum = op in (gr.GR_REDUCE_SUM, gr.GR_REDUCE_WSUM)
            x = xf if is_sum else xi
            weights = w if op == gr.GR_REDUCE_WSUM else None
            want = oracle.neighbor_reduce(r, c, op, x, w=weights)
            out = torch.full((n,), 9, dtype=torch.float64 if is_sum else torch.int32, device="cuda")
            gr.gr_neighbor_reduce(g, op, torch.from_numpy(x).cuda(), out)
            got = out.cpu().numpy()
            if is_sum:
                assert np.all(np.abs(got - want) <= sum_bound(r, c, x, weights)), op
            else:
                assert np.array_equal(got, want), op


@pytest.mark.parametrize("value", [np.inf, np.nan, -0.0])
def test_special_values_stay_in_their_rows(cuda_lib, value):
    import torch
    gr = cuda_lib
    n = 600
    r, c = csr([3, 300, 0, 5, 700, 1], n)
    x = np.ones(n)
    x[c[r[3]]] = value  # an entry of row 3
    want = np.array([x[c[r[v]:r[v + 1]]].sum() for v in range(n)])
    with gr.gr_graph_create(r, c) as g:
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        gr.gr_neighbor_reduce(g, gr.GR_REDUCE_SUM, torch.from_numpy(x).cuda(), out)
    got = out.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.array_equal(got[ok], want[ok])  # small integers and infinities: exact


@pytest.mark.parametrize("hubs,auths,deg", [(3, 5, 2), (64, 8, 4), (129, 67, 31), (2, 900, 450)])
def test_ranges_that_begin_inside_a_tile(cuda_lib, hubs, auths, deg):
    """HITS gathers the authorities' entries, which begin inside a tile."""
    import torch
    gr = cuda_lib
    links = {(h, hubs + (h * 7 + i * 3) % auths) for h in range(hubs) for i in range(deg)}
    n = hubs + auths
    both = sorted(links | {(b, a) for a, b in links})
    r = np.zeros(n + 1, np.int32)
    np.add.at(r, np.array([a for a, _ in both]) + 1, 1)
    r = np.cumsum(r).astype(np.int32)
    c = np.array([b for _, b in both], np.int32)
    with gr.gr_graph_create(r, c) as g:
        score = torch.empty(n, dtype=torch.float64, device="cuda")
        it = gr.gr_hits(g, hubs, score, max_iter=8, tol=0.0)
    want, _ = oracle.hits(r, c, hubs, it, 0.0)
    assert relative_l1(score.cpu().numpy(), want) <= 1e-10
