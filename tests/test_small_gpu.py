"""BFS of small graphs in one block: the largest and smallest sizes it takes,
frontiers of several chunks, long pull lists, its limits and its trace,
against the CPU oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import test_bfs_gpu as tb

pytestmark = pytest.mark.gpu


def from_pairs(n, pairs):
    """Symmetric CSR of an (k, 2) array of edges."""
    e = np.unique(np.concatenate([pairs, pairs[:, ::-1]]), axis=0)
    e = e[e[:, 0] != e[:, 1]]
    r = np.zeros(n + 1, np.int32)
    r[1:] = np.cumsum(np.bincount(e[:, 0], minlength=n))
    return r, e[:, 1].astype(np.int32)


def star_of_stars(n, hubs):
    """Vertex 0 joined to `hubs` vertices, the others shared out among them."""
    v = np.arange(1, n)
    return from_pairs(n, np.stack([np.where(v <= hubs, 0, 1 + (v % hubs)), v], 1))


def path_with_hub(n):
    """A path whose middle also has 20 leaves: maximum degree 22, n - 20 levels."""
    v = np.arange(n - 20)
    leaves = np.arange(n - 20, n)
    return from_pairs(n, np.concatenate([np.stack([v[:-1], v[1:]], 1),
                                         np.stack([np.full(20, n // 2), leaves], 1)]))


def lone_hub(n):
    """A hub with 3000 leaves out of the source's reach, and a random part."""
    rng = np.random.default_rng(n)
    part = rng.integers(3001, n, (6 * n, 2))
    return from_pairs(n, np.concatenate([np.stack([np.zeros(3000, int), np.arange(1, 3001)], 1),
                                         part]))


GRAPHS = {
    "stars_32768": lambda: star_of_stars(32768, 2000),
    "stars_32769": lambda: star_of_stars(32769, 2000),  # one too many: the grid
    "stars_31": lambda: star_of_stars(31, 17),
    "path_hub": lambda: path_with_hub(5000),
    "lone_hub": lambda: lone_hub(9000),
    "rmat_15": lambda: gg.rmat(15, 8, seed=3),
    "rmat_6": lambda: gg.rmat(6, 16, seed=3),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("direction", ["auto", "push"])
def test_depths_parents_and_trace(cuda_lib, name, direction):
    r, c = GRAPHS[name]()
    n = r.size - 1
    deg = np.diff(r)
    with cuda_lib.gr_graph_create(r, c) as g:
        for src in sorted({0, n - 1, int(np.argmax(deg)), int(np.argmin(deg))}):
            o = tb.opts(cuda_lib, direction)
            tb.check(cuda_lib, r, c, g, src, o)
            ref, _ = oracle.bfs(r, c, src)
            hist = np.bincount(ref[ref >= 0])
            tb.run_bfs(cuda_lib, g, src, o, with_parent=False)
            assert cuda_lib.gr_bfs_stats(g)[0] == len(hist)
            tr = cuda_lib.gr_bfs_trace(g)
            assert [f for _, f, _, _ in tr] == list(hist[:len(tr)])
            assert [e for _, _, e, _ in tr] == [int(deg[ref == l].sum()) for l in range(len(tr))]


def test_directed_and_level_cap(cuda_lib):
    r, c = path_with_hub(3000)
    # arcs only upwards
    up = np.repeat(np.arange(r.size - 1), np.diff(r)) < c
    rows = np.repeat(np.arange(r.size - 1), np.diff(r))[up]
    rd = np.zeros_like(r)
    rd[1:] = np.cumsum(np.bincount(rows, minlength=r.size - 1))
    cd = c[up]
    with cuda_lib.gr_graph_create(rd, cd) as g:
        for src in (0, 1500, 2999):
            tb.check(cuda_lib, rd, cd, g, src, symmetric=False)
    with cuda_lib.gr_graph_create(r, c) as g:
        with pytest.raises(cuda_lib.GrError) as ei:
            tb.run_bfs(cuda_lib, g, 0, cuda_lib.gr_opts(max_iters=9))
            cuda_lib.gr_bfs_stats(g)
        assert ei.value.status == cuda_lib.GR_ETIMEOUT
        tb.check(cuda_lib, r, c, g, 0)
