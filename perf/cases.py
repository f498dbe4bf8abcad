"""The framework's workloads as cases that can be timed and compared.

Each case is one call of a public entry point of `paper_1501_05387_gb300.gr`
on a graph that a user's program holds as a `Graph` handle: searches on
skewed and on mesh graphs, components, rankings, centrality and
neighbourhood reductions, from requests of a few thousand vertices to graphs
of millions. Graphs are built on the GPU from the seed alone, in the shapes
of this repository's generator: R-MAT (a, b, c = 0.57, 0.19, 0.19), with the
ids as the recursion gives them or renumbered at random, and 2D grids with
5 % of their edges deleted; weights are uniform in [1, wmax].
"""
import math

import torch

from paper_1501_05387_gb300 import gr

RMAT = (0.57, 0.19, 0.19)
GRID_DELETED = 0.05
DAMPING = 0.85
REDUCE = {"sum": gr.GR_REDUCE_SUM, "wsum": gr.GR_REDUCE_WSUM,
          "min": gr.GR_REDUCE_MIN, "max": gr.GR_REDUCE_MAX}


def listed():
    return [
        # a search on a small social graph: an interactive request, where
        # launches and latency are all there is
        {"name": "bfs_rmat_4k", "op": "bfs", "graph": "rmat", "n": 4096, "ef": 16},
        # the headline benchmark's graph: one search over 4.2 M vertices
        {"name": "bfs_rmat_4m", "op": "bfs", "graph": "rmat", "n": 1 << 22, "ef": 16},
        # hop counts on a road-like mesh: thousands of thin levels (the
        # serving pool's larger grid)
        {"name": "bfs_grid_1024", "op": "bfs", "graph": "grid", "side": 1024},
        # shortest paths on a skewed graph with the paper's weights, ids in
        # the arbitrary order that loaded datasets have
        {"name": "sssp_rmat_2m", "op": "sssp", "graph": "rmat", "n": 1 << 21, "ef": 16,
         "permute": True, "wmax": 64, "pred": False},
        # routing on a mesh, with the predecessor tree (serving pool's
        # smaller grid, an odd side)
        {"name": "sssp_grid_511", "op": "sssp", "graph": "grid", "side": 511, "wmax": 16,
         "pred": True},
        # routing from a batch of depots on a mesh
        {"name": "sssp_batch16_grid_300", "op": "sssp_batch", "graph": "grid", "side": 300,
         "wmax": 16, "k": 16},
        # 64 searches at once (landmarks, closeness samples)
        {"name": "bfs_batch64_rmat_1m", "op": "bfs_batch", "graph": "rmat", "n": 1 << 20,
         "ef": 16, "k": 64},
        # components of a skewed graph
        {"name": "cc_rmat_4m", "op": "cc", "graph": "rmat", "n": 1 << 22, "ef": 16},
        # a global ranking, a fixed number of iterations
        {"name": "pagerank_rmat_2m", "op": "pagerank", "graph": "rmat", "n": 1 << 21, "ef": 16,
         "iters": 20},
        # sampled betweenness centrality
        {"name": "bc64_rmat_256k", "op": "bc", "graph": "rmat", "n": 1 << 18, "ef": 16, "k": 64},
        # one aggregation over every neighbourhood (a feature or label sum),
        # ragged vertex count, arbitrary ids
        {"name": "reduce_sum_rmat_1500k", "op": "reduce", "graph": "rmat", "n": 1_500_001,
         "ef": 16, "permute": True, "reduce": "sum", "part": 1.0},
        # who-to-follow: hubs and authorities of a bipartite graph
        {"name": "hits_512k_128k", "op": "hits", "graph": "bipartite", "n": 1 << 19,
         "n_right": 1 << 17, "ef": 16, "iters": 20},
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["bfs", "bfs", "sssp", "sssp", "sssp_batch", "bfs_batch", "cc", "pagerank",
                     "bc", "reduce", "reduce", "hits", "salsa", "ppr"])
    case = {"op": op}
    grid = op == "sssp_batch" or (op in ("bfs", "sssp", "cc") and rng.random() < 0.4)
    if op in ("hits", "salsa"):
        case.update(graph="bipartite", n=_log_between(rng, 1 << 11, 1 << 19),
                    n_right=_log_between(rng, 1 << 10, 1 << 18), ef=rng.choice([8, 12, 16]))
    elif grid:
        case.update(graph="grid", side=_log_between(rng, 32, 256 if op == "sssp_batch" else 700))
    else:
        top = {"bc": 1 << 18, "bfs_batch": 1 << 19}.get(op, 1 << 21)
        case.update(graph="rmat", n=_log_between(rng, 1 << 11, top), ef=rng.choice([8, 12, 16]),
                    permute=rng.random() < 0.5)
        if op in ("bfs", "pagerank", "cc", "bfs_batch", "reduce"):
            case["directed"] = rng.random() < 0.25
    if op in ("sssp", "sssp_batch"):
        case["wmax"] = rng.choice([16, 64, 1000])
    if op == "sssp":
        case["pred"] = rng.random() < 0.5
    if op in ("sssp_batch", "bfs_batch", "bc"):
        case["k"] = rng.randint(2, 16 if op == "sssp_batch" else 64)
    if op in ("pagerank", "hits", "salsa", "ppr"):
        case["iters"] = rng.randint(5, 20)
    if op == "ppr":
        case["seeds"] = rng.randint(1, 16)
    if op == "reduce":
        case["reduce"] = rng.choice(["sum", "wsum", "min", "max"])
        case["part"] = rng.choice([1.0, 1.0, 0.3, 0.02])  # share of the vertices reduced
        if case["reduce"] == "wsum":
            case["wmax"] = 64
    return case


# ------------------------------------------------------------------- inputs

def _rmat_pairs(rows, cols, count, gen):
    """`count` R-MAT pairs (row, col) on `rows` x `cols` ids: the recursion's
    square scaled to those ranges."""
    bits = max(1, (max(rows, cols) - 1).bit_length())
    a, b, c = RMAT
    u = torch.zeros(count, dtype=torch.int32, device="cuda")
    v = torch.zeros(count, dtype=torch.int32, device="cuda")
    for _ in range(bits):
        r = torch.rand(count, device="cuda", generator=gen)
        down = r >= a + b
        u.mul_(2).add_(down)
        v.mul_(2).add_(torch.where(down, r >= a + b + c, r >= a))
    return (u.long() * rows) >> bits, (v.long() * cols) >> bits


def _csr(n, u, v):
    """Row offsets and columns (int32), rows sorted, duplicates removed."""
    key = torch.unique(u * n + v)
    row = torch.div(key, n, rounding_mode="floor")
    off = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return off, (key - row * n).int(), row


def _graph(case, seed):
    """(row_off, col, row of every entry, weights or None) of the case's graph."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["graph"] == "grid":
        side = case["side"]
        n = side * side
        at = torch.arange(n, device="cuda").view(side, side)
        u = torch.cat([at[:, :-1].reshape(-1), at[:-1].reshape(-1)])
        v = torch.cat([at[:, 1:].reshape(-1), at[1:].reshape(-1)])
        keep = torch.rand(u.numel(), device="cuda", generator=gen) >= GRID_DELETED
        u, v = u[keep], v[keep]
    elif case["graph"] == "bipartite":
        nl, nr = case["n"], case["n_right"]
        n = nl + nr
        u, v = _rmat_pairs(nl, nr, case["ef"] * max(nl, nr), gen)
        v = v + nl
    else:
        n = case["n"]
        u, v = _rmat_pairs(n, n, case["ef"] * n, gen)
        u, v = u[u != v], v[u != v]
    if case.get("permute"):
        p = torch.randperm(n, device="cuda", generator=gen)
        u, v = p[u], p[v]
    if not case.get("directed"):
        u, v = torch.cat([u, v]), torch.cat([v, u])
    off, col, row = _csr(n, u, v)
    w = None
    if "wmax" in case:
        # equal for both directions of an edge: a hash of its ends and the seed
        c = col.long()
        h = torch.minimum(row, c) * n + torch.maximum(row, c) + seed * 7_046_029_254_386_353
        h = (h ^ (h >> 31)) * 0x2545F4914F6CDD1D
        h = (h ^ (h >> 29)) * 0x5851F42D4C957F2D
        w = (((h >> 33) & 0x3FFFFFFF) % case["wmax"] + 1).int()
    return off, col, row, w


def _sources(off, k, seed):
    """k vertices with edges, from the seed."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1_000_003)
    some = torch.nonzero(off[1:] > off[:-1]).view(-1)
    return some[torch.randint(some.numel(), (k,), device="cuda", generator=gen)].cpu().numpy()


def _inputs(case, seed):
    """What the call takes besides the graph."""
    off, col, row, w = _graph(case, seed)
    n = off.numel() - 1
    s = {"off": off, "col": col, "row": row, "w": w, "n": n}
    op = case["op"]
    if op in ("bfs", "sssp"):
        s["src"] = int(_sources(off, 1, seed)[0])
    elif op in ("bfs_batch", "sssp_batch", "bc"):
        s["srcs"] = _sources(off, case["k"], seed)
    elif op == "ppr":
        s["srcs"] = sorted(set(_sources(off, case["seeds"], seed).tolist()))
    elif op == "reduce":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 2_000_003)
        if case["reduce"] in ("sum", "wsum"):
            s["x"] = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
            s["out"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        else:
            s["x"] = torch.randint(-2**31, 2**31 - 1, (n,), dtype=torch.int32, device="cuda",
                                   generator=gen)
            s["out"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["frontier"] = None
        if case["part"] < 1.0:
            pick = torch.randperm(n, device="cuda", generator=gen)
            s["frontier"] = pick[:max(1, int(n * case["part"]))].int()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["op"], s["case"] = case["op"], case
    s["g"] = gr.gr_graph_create(s["off"], s["col"], s["w"])
    n, op = s["n"], s["op"]
    if op in ("bfs", "sssp", "cc"):
        s["out"] = torch.empty(n, dtype=torch.int32, device="cuda")
    if op in ("bfs_batch", "sssp_batch"):
        s["out"] = torch.empty((case["k"], n), dtype=torch.int32, device="cuda")
    if op == "sssp":
        s["pred"] = torch.empty(n, dtype=torch.int32, device="cuda") if case["pred"] else None
    if op == "pagerank":
        s["out"] = torch.empty(n, dtype=torch.float32, device="cuda")
    if op in ("bc", "hits", "salsa", "ppr"):
        s["out"] = torch.empty(n, dtype=torch.float64, device="cuda")
    for k in ("off", "col", "row", "w"):
        del s[k]  # the handle holds its own copies
    return s


# --------------------------------------------------------------------- runs

def run(s):
    op, g, out, case = s["op"], s["g"], s["out"], s["case"]
    if op == "bfs":
        # hop counts only: a parent may be any vertex one level up, so parents
        # of two runs need not agree
        gr.gr_bfs(g, s["src"], out)
    elif op == "bfs_batch":
        gr.gr_bfs_batch(g, s["srcs"], out)
    elif op == "sssp":
        gr.gr_sssp(g, s["src"], out, s["pred"])
        if s["pred"] is not None:
            return {"dist": out, "pred": s["pred"]}
    elif op == "sssp_batch":
        gr.gr_sssp_batch(g, s["srcs"], out)
    elif op == "cc":
        return {"label": out, "components": gr.gr_cc(g, out)}
    elif op == "pagerank":
        gr.gr_pagerank(g, out, DAMPING, case["iters"], 0.0, count=False)
    elif op == "bc":
        gr.gr_bc(g, s["srcs"], out)
    elif op == "reduce":
        gr.gr_neighbor_reduce(g, REDUCE[case["reduce"]], s["x"], out, s["frontier"])
    elif op == "hits":
        gr.gr_hits(g, case["n"], out, case["iters"], 0.0, count=False)
    elif op == "salsa":
        gr.gr_salsa(g, case["n"], out, case["iters"], 0.0, count=False)
    elif op == "ppr":
        gr.gr_ppr(g, s["srcs"], out, DAMPING, case["iters"], 0.0, count=False)
    return out


def work(case):
    """Row offsets, columns (and weights) once, per-vertex inputs and outputs
    once; for an iterated ranking once per iteration. Of an R-MAT graph's
    pairs, duplicates and self-loops fall away: about 26 % of them at 4096
    vertices (19 % when directed), half that at every 16-fold size."""
    if case["graph"] == "grid":
        n = case["side"] ** 2
        m = 4 * n * (1 - GRID_DELETED)
    elif case["graph"] == "bipartite":
        n = case["n"] + case["n_right"]
        kept = 1 - 0.26 * (4096 / math.sqrt(case["n"] * case["n_right"])) ** 0.25
        m = 2 * kept * case["ef"] * max(case["n"], case["n_right"])
    else:
        n = case["n"]
        lost = (0.19 if case.get("directed") else 0.26) * (4096 / n) ** 0.25
        m = (1 if case.get("directed") else 2) * (1 - lost) * case["ef"] * n
    op, k, it = case["op"], case.get("k", 1), case.get("iters", 1)
    csr = 4 * (n + 1) + 4 * m
    wide = 4 * m if "wmax" in case else 0
    if op in ("bfs", "cc"):
        return {"bytes": csr + 4 * n, "flops": 0}
    if op == "sssp":
        return {"bytes": csr + wide + 4 * n * (2 if case["pred"] else 1), "flops": 0}
    if op == "bfs_batch":
        return {"bytes": csr + 4 * n * k, "flops": 0}
    if op == "sssp_batch":
        return {"bytes": csr + wide + 4 * n * k, "flops": 0}
    if op == "pagerank":
        return {"bytes": it * (csr + 8 * n), "flops": it * (m + 6.0 * n)}
    if op == "bc":
        # path counts and dependencies of every source: written once, read once
        return {"bytes": 2 * csr + 32 * n * k + 8 * n, "flops": 2.0 * m * k}
    if op == "reduce":
        el = 8 if case["reduce"] in ("sum", "wsum") else 4
        part = case["part"]
        return {"bytes": part * (csr + wide + el * n) + el * n, "flops": part * m}
    return {"bytes": it * (csr + 16 * n), "flops": it * (m + 6.0 * n)}


# -------------------------------------------------------------------- exact

def _gather(n, row, col, x, w=None):
    """Per row the sum of x[col] (times w)."""
    g = x[col] if w is None else x[col] * w
    return torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row, g)


def _pagerank(n, off, col, row, iters):
    deg = (off[1:] - off[:-1]).double()
    hang = deg == 0
    r = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        share = torch.where(hang, 0.0, r / deg.clamp(min=1.0))
        # rows point outwards: what vertex u gives goes to its columns
        into = torch.zeros_like(r).index_add_(0, col, share[row])
        r = (1 - DAMPING) / n + DAMPING * (into + r[hang].sum() / n)
    return r


def _ppr(n, off, col, row, seeds, iters):
    deg = (off[1:] - off[:-1]).double()
    hang = deg == 0
    t = torch.zeros(n, dtype=torch.float64, device="cuda")
    t[torch.tensor(seeds, device="cuda")] = 1.0 / len(seeds)
    r = t.clone()
    for _ in range(iters):
        share = torch.where(hang, 0.0, r / deg.clamp(min=1.0))
        r = (1 - DAMPING) * t + DAMPING * (_gather(n, row, col, share) + r[hang].sum() * t)
    return r


def _bipartite(n, n_left, off, col, row, iters, kind):
    deg = (off[1:] - off[:-1]).double()
    left = torch.arange(n, device="cuda") < n_left
    if kind == "hits":
        x = torch.where(left, 1.0 / math.sqrt(n_left), 0.0).double()
    else:
        x = torch.where(left & (deg > 0), 1.0, 0.0).double()
        x /= x.sum()
    for _ in range(iters):
        for side in (~left, left):
            y = _gather(n, row, col, x if kind == "hits" else x / deg.clamp(min=1.0))
            if kind == "hits":
                norm = y[side].norm()
                y = y / norm if norm > 0 else y
            x = torch.where(side, y, x)
    return x


def _bc(n, col, row, srcs):
    bc = torch.zeros(n, dtype=torch.float64, device="cuda")
    for s in srcs.tolist():
        depth = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        sigma = torch.zeros(n, dtype=torch.float64, device="cuda")
        depth[s], sigma[s] = 0, 1.0
        tree, level = [], 0
        while True:
            at = torch.nonzero((depth[row] == level) & (depth[col] < 0)).view(-1)
            if not at.numel():
                break
            r, c = row[at], col[at]
            depth[c] = level + 1
            sigma.index_add_(0, c, sigma[r])
            tree.append((r, c))
            level += 1
        delta = torch.zeros(n, dtype=torch.float64, device="cuda")
        for r, c in reversed(tree):
            delta.index_add_(0, r, sigma[r] / sigma[c] * (1.0 + delta[c]))
        delta[s] = 0.0
        bc += delta
    return bc


def exact(case, seed):
    """The floating results in 64 bits. Distances, hop counts, labels, minima
    and maxima are whole numbers, which have one right value."""
    op = case["op"]
    if op not in ("pagerank", "bc", "hits", "salsa", "ppr") and \
            not (op == "reduce" and case["reduce"] in ("sum", "wsum")):
        return None
    s = _inputs(case, seed)
    n, off, row = s["n"], s["off"], s["row"]
    col = s["col"].long()
    if op == "pagerank":
        return _pagerank(n, off, col, row, case["iters"])
    if op == "ppr":
        return _ppr(n, off, col, row, s["srcs"], case["iters"])
    if op in ("hits", "salsa"):
        return _bipartite(n, case["n"], off, col, row, case["iters"], op)
    if op == "bc":
        return _bc(n, col, row, s["srcs"])
    every = _gather(n, row, col, s["x"], s["w"].double() if case["reduce"] == "wsum" else None)
    if s["frontier"] is None:
        return every
    out = s["out"]  # entries outside the frontier stay as they were
    at = s["frontier"].long()
    out[at] = every[at]
    return out
