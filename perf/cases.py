"""Measured cases: the calls a program that clusters graphs with this package
makes, over the sizes, graph kinds and options it makes them with.

A case names a call path (``path``), a graph kind with its sizes, and the
options of the call. Graphs are drawn on the GPU from the seed: planted
partitions (block models, the well-clustered kind), road lattices (10% of the
lattice edges dropped, 1% diagonals, integer weights 1-10) and R-MAT
(0.57, 0.19, 0.19, 0.05), the kinds of the package's own generators.

The asynchronous mode (the default) makes concurrent moves in an order that
depends on timing, so its labels are a fixed answer only where the graph has
one: its cases are clear planted partitions of up to some 50,000 vertices, and
dense R-MAT graphs from about a million. Lattices, large planted partitions
and smaller R-MAT graphs, where many labellings score alike, run in the
deterministic mode, whose labels are reproducible; the two modes share the
schedule, the sweeps, the aggregation and the score.
"""
import math

import numpy as np
import torch

import paper_2312_13936_gb300 as lg


# ------------------------------------------------------------------ graphs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _csr(n, u, v, w=None):
    """Symmetric CSR of undirected edges: duplicates and self-loops dropped,
    targets ascending in every row (a duplicate's first weight stays)."""
    keep = u != v
    lo, hi = torch.minimum(u, v)[keep], torch.maximum(u, v)[keep]
    key = lo * n + hi
    if w is None:
        key = torch.unique(key)
        wt = None
    else:
        key, order = torch.sort(key, stable=True)
        wt = w[keep][order]
        first = torch.ones_like(key, dtype=torch.bool)
        first[1:] = key[1:] != key[:-1]
        key, wt = key[first], wt[first]
    lo, hi = torch.div(key, n, rounding_mode="floor"), key % n
    key = torch.cat([key, hi * n + lo])
    key, order = torch.sort(key)
    row = torch.div(key, n, rounding_mode="floor")
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    idx = (key - row * n).to(torch.int32)
    ww = torch.ones(idx.numel(), dtype=torch.float32, device="cuda") if wt is None else torch.cat([wt, wt])[order]
    return off, idx, ww


def _blocks_of(n, blocks):
    return torch.div(torch.arange(n, device="cuda") * blocks, n, rounding_mode="floor")


def _planted_edges(n, blocks, degree, mix, g):
    """Block model of near-equal contiguous blocks; a share mix of the edges
    leaves its block."""
    m = int(n * degree / 2)
    u = torch.randint(0, n, (m,), device="cuda", generator=g)
    b = torch.div(u * blocks, n, rounding_mode="floor")
    first = torch.div(b * n + blocks - 1, blocks, rounding_mode="floor")
    size = torch.div((b + 1) * n + blocks - 1, blocks, rounding_mode="floor") - first
    r = torch.rand(m, device="cuda", generator=g, dtype=torch.float64)
    inside = first + (r * size).long()
    outside = (first + size + (r * (n - size)).long()) % n
    return u, torch.where(torch.rand(m, device="cuda", generator=g) < mix, outside, inside)


def _road_edges(side, g):
    n = side * side
    at = torch.arange(n, device="cuda").view(side, side)
    u = torch.cat([at[:, :-1].reshape(-1), at[:-1, :].reshape(-1)])
    v = torch.cat([at[:, 1:].reshape(-1), at[1:, :].reshape(-1)])
    keep = torch.rand(u.numel(), device="cuda", generator=g) >= 0.1
    diag = torch.randint(0, (side - 1) * (side - 1), (2 * n // 100,), device="cuda", generator=g)
    diag = torch.div(diag, side - 1, rounding_mode="floor") * side + diag % (side - 1)
    u, v = torch.cat([u[keep], diag]), torch.cat([v[keep], diag + side + 1])
    return u, v, torch.randint(1, 11, (u.numel(),), device="cuda", generator=g).float()


def _rmat_edges(n, edge_factor, g):
    """R-MAT (0.57, 0.19, 0.19, 0.05) on the smallest scale that holds n
    vertices, its ids folded onto [0, n) when n is no power of two."""
    m = n * edge_factor
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(max(1, (n - 1).bit_length())):
        r = torch.rand(m, device="cuda", generator=g)
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return u % n, v % n


def _edges(case, g):
    if case["graph"] == "planted":
        return _planted_edges(case["n"], case["blocks"], case["degree"], case["mix"], g) + (None,)
    if case["graph"] == "road":
        return _road_edges(math.isqrt(case["n"]), g)
    return _rmat_edges(case["n"], case["degree"], g) + (None,)


def _graph(case, g):
    return _csr(case["n"], *_edges(case, g))


def _entries(case):
    """CSR entries of a case's graph, about (duplicates aside)."""
    return int(case["n"] * (3.64 if case["graph"] == "road" else case["degree"] * (2 if case["graph"] == "rmat" else 1)))


def _edge_list(case, g):
    """An edge list as it arrives, in no order: n * degree different R-MAT
    edges, an eighth of them again the other way round, and some self-loops."""
    n, m = case["n"], case["n"] * case["degree"]
    u, v = _rmat_edges(n, 3 * case["degree"], g)
    key = torch.unique((torch.minimum(u, v) * n + torch.maximum(u, v))[u != v])
    key = key[torch.randperm(key.numel(), device="cuda", generator=g)[:m]]
    u, v = torch.div(key, n, rounding_mode="floor"), key % n
    src, dst = torch.cat([u, v[:m // 8], u[:m // 64]]), torch.cat([v, u[:m // 8], u[:m // 64]])
    order = torch.randperm(src.numel(), device="cuda", generator=g)
    src, dst = src[order], dst[order]
    w = torch.randint(1, 11, (src.numel(),), device="cuda", generator=g).float() if case["weighted"] else None
    return src, dst, w


def _ladder(graphs, lo, hi):
    """Sizes spread evenly over the logarithm of [lo, hi]."""
    return [round(lo * (hi / lo) ** (k / max(1, graphs - 1))) for k in range(graphs)]


def _union(case, g):
    """The graphs of a batch as one segmented CSR: block models whose sizes
    climb from 100 vertices to n, 4-64 blocks, mean degree 8-32; indices
    local to each graph."""
    sizes = _ladder(case["graphs"], 100, case["n"])
    seg = np.zeros(len(sizes) + 1, dtype=np.int64)
    seg[1:] = np.cumsum(sizes)
    us, vs = [], []
    for k, n in enumerate(sizes):
        blocks = min(4 + (7 * k) % 61, n // 8)
        u, v = _planted_edges(n, blocks, 8 + (5 * k) % 25, 0.3, g)
        us.append(u + int(seg[k]))
        vs.append(v + int(seg[k]))
    off, idx, w = _csr(int(seg[-1]), torch.cat(us), torch.cat(vs))
    start = torch.from_numpy(seg).cuda()
    row = torch.repeat_interleave(torch.arange(off.numel() - 1, device="cuda"), off[1:] - off[:-1])
    own = torch.searchsorted(start, row, right=True) - 1
    return seg, off, (idx - start[own]).to(torch.int32), w


def _pool(case):
    """The graphs of a serving mix: block models from 1000 to n vertices and,
    every fourth, an R-MAT graph of 4096 vertices and more."""
    pool = []
    for k, n in enumerate(_ladder(case["graphs"], 1000, case["n"])):
        if k % 4 == 3:
            pool.append({"graph": "rmat", "n": 4096 << min(3, k // 4), "degree": 16})
        else:
            pool.append({"graph": "planted", "n": n, "blocks": 10 + k, "degree": 16, "mix": 0.2})
    return pool


def _tiles(n, tile):
    """Labels of a lattice's tile x tile squares."""
    side = math.isqrt(n)
    at = torch.arange(side, device="cuda") // tile
    per = (side + tile - 1) // tile
    return (at[:, None] * per + at[None, :]).reshape(-1).to(torch.int32)


def _score64(off, idx, w, labels):
    """Eq. 1 in 64 bits."""
    n = off.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    lab, w = labels.long(), w.double()
    two_m = w.sum()
    inside = w[lab[row] == lab[idx.long()]].sum()
    k = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, lab[row], w)
    return float(inside / two_m - (k * k).sum() / (two_m * two_m))


# ------------------------------------------------------------------- cases
def listed():
    return [
        # a program that clusters each small graph it meets once: upload, run, release
        {"name": "once_planted_2k", "path": "once", "graph": "planted", "n": 2000, "blocks": 10, "degree": 24,
         "mix": 0.1, "validate": True},
        # a resident graph clustered again and again with the defaults: small
        {"name": "run_planted_10k", "path": "run", "mode": "async", "graph": "planted", "n": 10007, "blocks": 16,
         "degree": 32, "mix": 0.1, "louvain": False},
        # and the middle of the planted range
        {"name": "run_planted_50k", "path": "run", "mode": "async", "graph": "planted", "n": 50000, "blocks": 16,
         "degree": 32, "mix": 0.1, "louvain": False},
        # reproducible labels on a social-network-like graph of the tuned class
        {"name": "det_planted_200k", "path": "run", "mode": "det", "graph": "planted", "n": 200000, "blocks": 64,
         "degree": 24, "mix": 0.3, "louvain": False},
        # road networks: a city's, and the largest of the benchmark (5000 x 5000)
        {"name": "det_road_1m", "path": "run", "mode": "det", "graph": "road", "n": 1000 * 1000, "louvain": False},
        {"name": "det_road_25m", "path": "run", "mode": "det", "graph": "road", "n": 5000 * 5000, "louvain": False},
        # heavy-tailed web-like graphs: small and sparse, and large and dense
        {"name": "det_rmat_64k", "path": "run", "mode": "det", "graph": "rmat", "n": 1 << 16, "degree": 16,
         "louvain": False},
        {"name": "run_rmat_1m", "path": "run", "mode": "async", "graph": "rmat", "n": 1 << 20, "degree": 56,
         "louvain": False},
        # many graphs in one call
        {"name": "batch_256", "path": "batch", "graphs": 256, "n": 20000},
        # requests served from host memory with continuous batching
        {"name": "serve_16", "path": "serve", "graphs": 16, "n": 60000},
        # an edge list turned into the graph it describes
        {"name": "edges_rmat_1m", "path": "edges", "graph": "rmat", "n": 1 << 20, "degree": 40, "weighted": False,
         "combine": "sum"},
        # a given labelling scored and checked (Eq. 1, disconnected communities)
        {"name": "score_road_9m", "path": "score", "graph": "road", "n": 3000 * 3000, "tile": 40},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ones' ranges."""
    path = rng.choice(["once", "run", "run", "run", "run", "run", "run", "batch", "serve", "edges", "score"])
    if path == "once":
        n = _log(rng, 300, 4000)
        return {"path": path, "graph": "planted", "n": n, "blocks": rng.randint(4, 10), "degree": rng.randint(24, 32),
                "mix": round(rng.uniform(0.05, 0.15), 3), "validate": rng.random() < 0.5}
    if path == "batch":
        return {"path": path, "graphs": _log(rng, 8, 256), "n": _log(rng, 2000, 20000)}
    if path == "serve":
        return {"path": path, "graphs": rng.randint(4, 16), "n": _log(rng, 4000, 60000)}
    if path == "edges":
        return {"path": path, "graph": "rmat", "n": _log(rng, 2000, 1 << 20), "degree": rng.randint(4, 32),
                "weighted": rng.random() < 0.5, "combine": rng.choice(["sum", "max"])}
    if path == "score":
        return {"path": path, "graph": "road", "n": _log(rng, 60, 3000) ** 2, "tile": rng.randint(10, 80)}
    kind = rng.choice(["planted", "planted", "planted", "road", "rmat", "rmat"])
    case = {"path": path, "mode": "det", "graph": kind, "louvain": rng.random() < 0.125}
    if kind == "road":
        return {**case, "n": _log(rng, 100, 4999) ** 2}
    if kind == "rmat":
        if rng.random() < 0.33:
            return {**case, "mode": "async", "n": rng.randint(950000, 1040000), "degree": rng.randint(50, 56)}
        return {**case, "n": _log(rng, 4096, 100000), "degree": rng.randint(8, 24)}
    if rng.random() < 0.67:
        return {**case, "mode": "async", "n": _log(rng, 2000, 50000), "blocks": 16, "degree": 32,
                "mix": round(rng.uniform(0.05, 0.12), 3)}
    return {**case, "n": _log(rng, 5000, 200000), "blocks": rng.randint(8, 64), "degree": rng.randint(8, 24),
            "mix": round(rng.uniform(0.1, 0.4), 3)}


def prepare(case, seed):
    g = _generator(seed)
    path = case["path"]
    if path == "batch":
        seg, off, idx, w = _union(case, g)
        return {"path": path, "handle": lg.LeidenBatch(seg, off, idx, w)}
    if path == "serve":
        pool = []
        for c in _pool(case):
            pool.append(tuple(t.cpu().numpy() for t in _graph(c, g)))
        vertices, entries = sum(len(p[0]) - 1 for p in pool), sum(len(p[1]) for p in pool)
        server = lg.LeidenServer(vertices, entries, max_graphs=len(pool), mode=lg.LEIDEN_DETERMINISTIC)
        return {"path": path, "pool": pool, "server": server}
    if path == "edges":
        src, dst, w = _edge_list(case, g)
        return {"path": path, "n": case["n"], "src": src.to(torch.int32), "dst": dst.to(torch.int32), "w": w,
                "combine": case["combine"]}
    off, idx, w = _graph(case, g)
    if path == "once":
        return {"path": path, "graph": (off, idx, w), "validate": case["validate"]}
    if path == "score":
        return {"path": path, "graph": (off, idx, w), "labels": _tiles(case["n"], case["tile"])}
    mode = lg.LEIDEN_DETERMINISTIC if case["mode"] == "det" else lg.LEIDEN_ASYNC
    return {"path": path, "handle": lg.Leiden(off, idx, w), "mode": mode,
            "flags": lg.FLAG_LOUVAIN if case["louvain"] else 0}


def run(state):
    path = state["path"]
    if path == "run":
        labels, q, stats = state["handle"].run(mode=state["mode"], flags=state["flags"])
        return {"labels": labels, "q": q, "communities": stats.communities}
    if path == "once":
        handle = lg.Leiden(*state["graph"], validate=state["validate"])
        labels, q, stats = handle.run()
        handle.close()
        return {"labels": labels, "q": q, "communities": stats.communities}
    if path == "batch":
        labels, q, stats = state["handle"].run(mode=lg.LEIDEN_DETERMINISTIC)
        return {"labels": labels, "q": q, "communities": state["handle"].info()[1]}
    if path == "serve":
        server, done = state["server"], []
        for off, idx, w in state["pool"]:
            server.submit(off, idx, w)
        while len(done) < len(state["pool"]):
            server.step()
            done += server.results()
        done.sort(key=lambda r: r[0])
        return {"labels": np.concatenate([r[1] for r in done]), "q": np.array([r[2] for r in done]),
                "communities": np.array([r[4] for r in done])}
    if path == "edges":
        off, idx, w = lg.csr_from_edges(state["n"], state["src"], state["dst"], state["w"], drop_self_loops=True,
                                        combine=state["combine"])
        return {"offsets": off, "indices": idx, "weights": w}
    off, idx, w = state["graph"]
    return {"q": lg.modularity(off, idx, w, state["labels"]),
            "disconnected": lg.disconnected(off, idx, state["labels"])}


def work(case):
    """The graph read once (offsets 8 bytes a vertex, index and weight 8 bytes
    an entry) and the labels written once; an edge list read once and its
    graph written once."""
    path = case["path"]
    if path == "batch":
        sizes = _ladder(case["graphs"], 100, case["n"])
        n, m = sum(sizes), sum(s * (8 + (5 * k) % 25) for k, s in enumerate(sizes))
    elif path == "serve":
        n, m = sum(c["n"] for c in _pool(case)), sum(_entries(c) for c in _pool(case))
    else:
        n, m = case["n"], _entries(case)
    if path == "edges":
        listed_edges = (m // 2) * 73 // 64
        return {"bytes": listed_edges * (12 if case["weighted"] else 8) + 8 * n + 8 * m, "flops": 0}
    return {"bytes": 8 * n + 8 * m + 4 * n, "flops": 2 * m}


def exact(case, seed):
    """In 64 bits: the score of the planted blocks, which the asynchronous
    runs recover, the score of a given labelling, the merged weights of an
    edge list. A deterministic run's labels have no closed form."""
    path = case["path"]
    g = _generator(seed)
    if path == "once" or (path == "run" and case["mode"] == "async" and case["graph"] == "planted"):
        q = _score64(*_graph(case, g), _blocks_of(case["n"], case["blocks"]))
        return {"labels": None, "q": q, "communities": None}
    if path == "score":
        return {"q": _score64(*_graph(case, g), _tiles(case["n"], case["tile"])), "disconnected": None}
    if path != "edges":
        return None
    n = case["n"]
    u, v, w = _edge_list(case, g)
    w = torch.ones(u.numel(), dtype=torch.float64, device="cuda") if w is None else w.double()
    u, v, w = u[u != v], v[u != v], w[u != v]
    key, at = torch.unique(torch.cat([u * n + v, v * n + u]), return_inverse=True)
    w = torch.cat([w, w])
    if case["combine"] == "max":
        out = torch.zeros(key.numel(), dtype=torch.float64, device="cuda").scatter_reduce_(0, at, w, "amax")
    else:
        out = torch.zeros(key.numel(), dtype=torch.float64, device="cuda").index_add_(0, at, w)
    row = torch.div(key, n, rounding_mode="floor")
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return {"offsets": off, "indices": key % n, "weights": out}
