"""The workloads this library is timed on: PageRank (pull, push, batched, personalised), BFS,
betweenness centrality and SpMV over skewed, uniform and grid graphs, through the Python entry
points.  Graphs are drawn here with torch alone, from the seed alone.

A case is a dict: ``kind`` (what is called), ``graph`` ("rmat", "er" or "grid"), its size, and the
options of the call.  R-MAT and uniform graphs take any vertex count; a grid is side x side.
"""
from __future__ import annotations

import math

import torch

import paper_1904_02241_gb300 as T

DAMPING = 0.85
ITERS = 20
EDGE_FACTOR = 16
RMAT_ABC = (0.57, 0.19, 0.19)
GRID_DROP = 0.05
CHUNK = 1 << 26      # edges drawn at a time


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------

def listed():
    return [
        # A small graph ranked again and again (a service, a test): launches and latency count.
        {"name": "pull_small", "kind": "pull", "graph": "rmat", "V": 1 << 16, "blocks": 4, "order": "natural"},
        # The headline: a large social graph, blocks of one CTA's shared memory, renumbered.
        {"name": "pull_rmat", "kind": "pull", "graph": "rmat", "V": 1 << 24, "blocks": 0, "order": "outdegree"},
        # No skew and no locality, ragged size, the paper's source ranges: the most partial sums.
        {"name": "pull_uniform", "kind": "pull", "graph": "er", "V": 6000011, "blocks": 0, "order": "natural"},
        # The push variant (Alg. 5), default sums and default blocks.
        {"name": "push_rmat", "kind": "push", "graph": "rmat", "V": 1 << 22, "blocks": 0},
        # Hop levels of a social graph from a few sources, direction-optimised.
        {"name": "bfs_rmat", "kind": "bfs", "graph": "rmat", "V": 1 << 22, "sources": 4, "mode": "diropt"},
        # The same on a road-like graph: thousands of levels, each with a small frontier.
        {"name": "bfs_grid", "kind": "bfs", "graph": "grid", "side": 2048, "sources": 1, "mode": "diropt"},
        # The topology-driven pull BFS of the paper, blocked in every level, ragged size.
        {"name": "bfs_pull", "kind": "bfs", "graph": "rmat", "V": 5000003, "sources": 2, "mode": "pull"},
        # Personalised ranks of 256 users in one batch.
        {"name": "ppr_batch", "kind": "ppr", "graph": "rmat", "V": 1 << 22, "columns": 256},
        # A thousand independent small graphs in one launch.
        {"name": "many_graphs", "kind": "multi", "graphs": 1000, "lo": 10, "hi": 16},
        # A sparse matrix (skewed rows) times a vector, column blocks.
        {"name": "spmv", "kind": "spmv", "graph": "rmat", "V": 1 << 22, "blocks": 8},
        # Betweenness scores from a few sources: a forward and a backward sweep each.
        {"name": "bc", "kind": "bc", "graph": "rmat", "V": 1 << 18, "sources": 4},
        # One ranking job from host buffers: load, transpose, renumber, cut, iterate, read back.
        {"name": "job", "kind": "job", "graph": "rmat", "V": 1 << 22, "blocks": 0, "order": "outdegree"},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pull", "pull", "push", "bfs", "bfs_grid", "ppr", "multi", "spmv", "bc", "job"])
    if kind == "pull":
        graph = rng.choice(["rmat", "rmat", "er"])
        V = _size(rng, 1 << 14, 12000000)
        if V < 1 << 18:
            return {"kind": "pull", "graph": graph, "V": V, "blocks": rng.choice([2, 4, 8]), "order": "natural"}
        return {"kind": "pull", "graph": graph, "V": V, "blocks": 0, "order": rng.choice(["natural", "outdegree"])}
    if kind == "push":
        return {"kind": "push", "graph": rng.choice(["rmat", "er"]), "V": _size(rng, 1 << 15, 1 << 23), "blocks": 0}
    if kind == "bfs":
        return {"kind": "bfs", "graph": "rmat", "V": _size(rng, 1 << 15, 6000000), "sources": rng.randint(1, 4),
                "mode": rng.choice(["diropt", "diropt", "pull"])}
    if kind == "bfs_grid":
        return {"kind": "bfs", "graph": "grid", "side": _size(rng, 200, 2048), "sources": 1, "mode": "diropt"}
    if kind == "ppr":
        return {"kind": "ppr", "graph": "rmat", "V": _size(rng, 1 << 14, 3000000), "columns": _size(rng, 5, 256)}
    if kind == "multi":
        lo = rng.randint(8, 12)
        return {"kind": "multi", "graphs": _size(rng, 40, 600), "lo": lo, "hi": rng.randint(lo, 15)}
    if kind == "spmv":
        return {"kind": "spmv", "graph": rng.choice(["rmat", "er"]), "V": _size(rng, 1 << 16, 1 << 23),
                "blocks": rng.choice([4, 8, 16])}
    if kind == "bc":
        return {"kind": "bc", "graph": "rmat", "V": _size(rng, 1 << 14, 1 << 21), "sources": rng.randint(1, 4)}
    return {"kind": "job", "graph": "rmat", "V": _size(rng, 1 << 18, 1 << 23), "blocks": 0, "order": "outdegree"}


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------

def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _rmat_chunk(gen, levels, n):
    """n edge draws, each descending ``levels`` quadrant levels."""
    a, b, c = RMAT_ABC
    s = torch.zeros(n, dtype=torch.int32, device="cuda")
    d = torch.zeros(n, dtype=torch.int32, device="cuda")
    for _ in range(levels):
        u = torch.rand(n, generator=gen, device="cuda")
        s = s * 2 + (u >= a + b)
        d = d * 2 + (((u >= a) & (u < a + b)) | (u >= a + b + c))
    return s.long(), d.long()


def _draw_edges(case, gen):
    """Directed (source, destination) draws of the case's graph, repeats included."""
    if case["graph"] == "grid":
        n = case["side"]
        v = torch.arange(n * n, device="cuda").reshape(n, n)
        u = torch.cat([v[:, :-1].reshape(-1), v[:-1].reshape(-1)])
        w = torch.cat([v[:, 1:].reshape(-1), v[1:].reshape(-1)])
        keep = torch.rand(u.numel(), generator=gen, device="cuda") >= GRID_DROP
        return u[keep], w[keep]
    V = case["V"]
    M = EDGE_FACTOR * V
    ss, ds = [], []
    for start in range(0, M, CHUNK):
        n = min(CHUNK, M - start)
        if case["graph"] == "er":
            ss.append(torch.randint(V, (n,), generator=gen, device="cuda"))
            ds.append(torch.randint(V, (n,), generator=gen, device="cuda"))
        else:
            s, d = _rmat_chunk(gen, (V - 1).bit_length(), n)
            ss.append(s)
            ds.append(d)
    s, d = torch.cat(ss), torch.cat(ds)
    if case["graph"] == "rmat":  # relabel (no locality in the ids), folded onto V vertices
        perm = torch.randperm(1 << (V - 1).bit_length(), generator=gen, device="cuda") % V
        s, d = perm[s], perm[d]
    return s, d


def _csr(V, s, d):
    """Out-edge CSR (int32) without self loops and repeated edges, rows sorted."""
    key = (s * V + d)[s != d]
    del s, d
    key = torch.unique(key)
    s = torch.div(key, V, rounding_mode="floor")
    rowptr = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(s, minlength=V), 0)
    return rowptr.to(torch.int32), (key - s * V).to(torch.int32)


def _vertices(case):
    return case["side"] ** 2 if case["graph"] == "grid" else case["V"]


def _graph(case, gen):
    V = _vertices(case)
    s, d = _draw_edges(case, gen)
    if case["kind"] in ("bfs", "bc"):  # undirected
        s, d = torch.cat([s, d]), torch.cat([d, s])
    return (V, *_csr(V, s, d))


def _sources(rowptr, count, gen):
    cand = torch.nonzero(rowptr[1:] > rowptr[:-1]).reshape(-1)
    pick = torch.randint(cand.numel(), (count,), generator=gen, device="cuda")
    return cand[pick].tolist()


def _batch(case, gen):
    """A batch of R-MAT graphs, scales lo to hi equally often and in random order: the union's CSR
    and vertex offsets."""
    n, lo, hi = case["graphs"], case["lo"], case["hi"]
    scale = lo + torch.randperm(n, generator=gen, device="cuda") % (hi + 1 - lo)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.ones_like(scale) << scale, 0)
    ss, ds = [], []
    for sc in range(lo, hi + 1):
        base = off[:-1][scale == sc]
        if base.numel() == 0:
            continue
        V = 1 << sc
        s, d = _rmat_chunk(gen, sc, base.numel() * EDGE_FACTOR * V)
        which = torch.arange(base.numel(), device="cuda").repeat_interleave(EDGE_FACTOR * V)
        perm = torch.argsort(torch.rand((base.numel(), V), generator=gen, device="cuda"), dim=1).reshape(-1)
        ss.append(perm[which * V + s] + base[which])
        ds.append(perm[which * V + d] + base[which])
    V = int(off[-1])
    return (V, *_csr(V, torch.cat(ss), torch.cat(ds)), off)


def _inputs(case, seed):
    """Everything drawn from the seed: the graph and what goes with it."""
    gen = _rng(seed)
    x = {}
    if case["kind"] == "multi":
        x["V"], x["rowptr"], x["colidx"], x["off"] = _batch(case, gen)
        return x
    x["V"], x["rowptr"], x["colidx"] = _graph(case, gen)
    if case["kind"] in ("bfs", "bc"):
        x["sources"] = _sources(x["rowptr"], case["sources"], gen)
    elif case["kind"] == "ppr":
        x["sources"] = _sources(x["rowptr"], case["columns"], gen)
    elif case["kind"] == "spmv":
        x["vals"] = torch.rand(x["colidx"].numel(), generator=gen, device="cuda") * 2 - 1
        x["x"] = torch.randn(x["V"], generator=gen, device="cuda")
    return x


# ------------------------------------------------------------------------------------------
# preparing, running
# ------------------------------------------------------------------------------------------

def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "multi":
        st["M"] = T.multigraph_load(x["rowptr"], x["colidx"], x["off"].to(torch.int32))
        st["out"] = torch.empty(x["V"], dtype=torch.float32, device="cuda")
        return st
    if kind == "job":
        st["case"] = case
        st["rowptr"], st["colidx"] = x["rowptr"].cpu().pin_memory(), x["colidx"].cpu().pin_memory()
        st["out"] = torch.empty(x["V"], dtype=torch.float32).pin_memory()
        return st
    G = st["G"] = T.graph_load_csr(x["rowptr"], x["colidx"], V=x["V"])
    if kind == "pull":
        st["P"] = T.tocab_partition(G, T.TC_PULL, case["blocks"], block_policy="smem", order=case["order"])
    elif kind == "push":
        st["P"] = T.tocab_partition(G, T.TC_PUSH, case["blocks"])
    elif kind == "bfs":
        st["sources"] = x["sources"]
        st["pull"] = case["mode"] == "pull"
        st["P"] = T.tocab_partition(G, T.TC_PULL, 8, smem_stage=-1) if st["pull"] else None
    elif kind == "bc":
        st["sources"] = x["sources"]
    elif kind == "ppr":
        st["sources"] = x["sources"]
        T.ppr_set_tuning(G, hot=-1, tile=0 if case["columns"] > 64 else 32)
        st["out"] = torch.empty((x["V"], case["columns"]), dtype=torch.float32, device="cuda")
    elif kind == "spmv":
        st["x"] = x["x"]
        st["P"] = T.tocab_partition(G, T.TC_PUSH, case["blocks"], merge_range=8192)
        T.part_set_values(st["P"], x["vals"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "pull":
        return T.pagerank_pull(st["G"], st["P"], damping=DAMPING, iters=ITERS)
    if kind == "push":
        return T.pagerank_push(st["G"], st["P"], damping=DAMPING, iters=ITERS)
    if kind == "bfs":
        if st["pull"]:
            return [T.bfs_pull(st["G"], st["P"], s, tocab_threshold=0.0) for s in st["sources"]]
        return [T.bfs_pull(st["G"], None, s, tocab_threshold=-1.0, push_threshold=1.0 / 24) for s in st["sources"]]
    if kind == "ppr":
        return T.ppr_batch(st["G"], st["sources"], damping=DAMPING, iters=ITERS, out=st["out"])
    if kind == "multi":
        return T.pagerank_multi(st["M"], damping=DAMPING, iters=ITERS, out=st["out"],
                                lanes_per_vertex=T.TC_MULTI_RESIDENT)
    if kind == "spmv":
        return T.spmv_tocab(st["P"], st["x"])
    if kind == "bc":
        return T.bc(st["G"], st["sources"])
    G = T.graph_load_csr(st["rowptr"], st["colidx"])
    P = T.tocab_partition(G, T.TC_PULL, st["case"]["blocks"], block_policy="smem", order=st["case"]["order"])
    T.pagerank_pull(G, P, damping=DAMPING, iters=ITERS, out=st["out"])
    P.free()
    G.free()
    return st["out"]


# ------------------------------------------------------------------------------------------
# the work of a pass
# ------------------------------------------------------------------------------------------

def _edges(graph, V):
    """Expected number of distinct edges (int)."""
    M = EDGE_FACTOR * V
    if graph == "er":
        return int(V * V * -math.expm1(-M / (V * V)))
    L = (V - 1).bit_length()
    a, b, c = RMAT_ABC
    d = 1 - a - b - c
    total = 0.0
    for i in range(L + 1):              # i levels in quadrant a, j in b or c, the rest in d
        for j in range(L + 1 - i):
            cells = math.comb(L, i) * math.comb(L - i, j) * 2.0 ** j
            total += cells * -math.expm1(-M * a ** i * b ** j * d ** (L - i - j))
    return int(total)


def work(case):
    kind = case["kind"]
    if kind == "multi":
        scales = range(case["lo"], case["hi"] + 1)
        V = case["graphs"] * sum(1 << s for s in scales) // len(scales)
        E = case["graphs"] * sum(_edges("rmat", 1 << s) for s in scales) // len(scales)
    else:
        V = _vertices(case)
        E = int((1 - GRID_DROP) * 4 * V) if case["graph"] == "grid" else _edges(case["graph"], V)
    if kind in ("pull", "push", "multi"):   # the CSR, out-degree reciprocals, ranks in and out
        return {"bytes": ITERS * (4 * E + 16 * V), "flops": ITERS * (E + 4 * V)}
    if kind == "job":                       # the same, and the CSR and the ranks over the host link
        return {"bytes": ITERS * (4 * E + 16 * V) + 4 * E + 8 * V, "flops": ITERS * (E + 4 * V)}
    if kind == "ppr":                       # the CSR and the rank matrix in and out
        n = case["columns"]
        return {"bytes": ITERS * (4 * E + 8 * V + 8 * V * n), "flops": ITERS * 2 * E * n}
    if kind == "spmv":                      # columns, values, row offsets, x, y
        return {"bytes": 8 * E + 12 * V, "flops": 2 * E}
    if case["graph"] != "grid":
        E *= 2
    if kind == "bfs":                       # the CSR, levels out
        return {"bytes": case["sources"] * (4 * E + 8 * V), "flops": 0}
    # bc: forward (CSR in, depth and sigma out) and backward (CSR, depth, sigma in, scores out)
    return {"bytes": case["sources"] * (8 * E + 40 * V), "flops": case["sources"] * 3 * E}


# ------------------------------------------------------------------------------------------
# the same outputs in 64 bits, by plain torch
# ------------------------------------------------------------------------------------------

def _rows(rowptr):
    deg = (rowptr[1:] - rowptr[:-1]).long()
    return torch.repeat_interleave(torch.arange(deg.numel(), device="cuda"), deg), deg


def _gather_add(V, index, values):
    return torch.zeros(V, dtype=torch.float64, device="cuda").index_add_(0, index, values)


def _exact_pagerank(x):
    """Alg. 1 with the dangling mass spread over the vertices of its own graph."""
    V = x["V"]
    src, deg = _rows(x["rowptr"])
    dst = x["colidx"].long()
    inv = torch.where(deg > 0, 1.0 / deg.double(), 0.0)
    off = x.get("off", torch.tensor([0, V], device="cuda"))
    size = off[1:] - off[:-1]
    gid = torch.repeat_interleave(torch.arange(size.numel(), device="cuda"), size)
    n = size.double()[gid]
    r = 1.0 / n
    for _ in range(ITERS):
        D = torch.zeros(size.numel(), dtype=torch.float64, device="cuda")
        D.index_add_(0, gid, torch.where(deg > 0, 0.0, r))
        r = (1 - DAMPING) / n + DAMPING * (_gather_add(V, dst, (r * inv)[src]) + D[gid] / n)
    return r


def _exact_ppr(x):
    """Column j: teleport and dangling mass to source j."""
    V, n = x["V"], len(x["sources"])
    src, deg = _rows(x["rowptr"])
    inv = torch.where(deg > 0, 1.0 / deg.double(), 0.0)
    order = torch.argsort(x["colidx"].long() * V + src)     # in-edges, by destination
    in_ptr = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    in_ptr[1:] = torch.cumsum(torch.bincount(x["colidx"].long(), minlength=V), 0)
    A = torch.sparse_csr_tensor(in_ptr, src[order], inv[src[order]], (V, V))
    out = torch.empty((V, n), dtype=torch.float64, device="cuda")
    for j0 in range(0, n, 32):
        s = torch.tensor(x["sources"][j0:j0 + 32], device="cuda")
        j = torch.arange(s.numel(), device="cuda")
        r = torch.zeros((V, s.numel()), dtype=torch.float64, device="cuda")
        r[s, j] = 1.0
        for _ in range(ITERS):
            D = (r * (deg == 0).double()[:, None]).sum(0)
            r = DAMPING * (A @ r)
            r[s, j] += (1 - DAMPING) + DAMPING * D
        out[:, j0:j0 + 32] = r
    return out


def _exact_levels(x, source):
    V = x["V"]
    rowptr, colidx = x["rowptr"].long(), x["colidx"].long()
    level = torch.full((V,), -1, dtype=torch.int32, device="cuda")
    front = torch.tensor([source], device="cuda")
    depth = 0
    while front.numel():
        level[front] = depth
        deg = rowptr[front + 1] - rowptr[front]
        first = torch.repeat_interleave(rowptr[front] - torch.cumsum(deg, 0) + deg, deg)
        nbr = colidx[first + torch.arange(first.numel(), device="cuda")]
        front = torch.unique(nbr[level[nbr] < 0])
        depth += 1
    return level


def _exact_bc(x):
    V = x["V"]
    src, _ = _rows(x["rowptr"])
    dst = x["colidx"].long()
    score = torch.zeros(V, dtype=torch.float64, device="cuda")
    for s in x["sources"]:
        level = _exact_levels(x, s)
        tree = (level[src] >= 0) & (level[dst] == level[src] + 1)   # edges on shortest paths
        u, w = src[tree], dst[tree]
        lu = level[u]
        sigma = torch.zeros(V, dtype=torch.float64, device="cuda")
        sigma[s] = 1.0
        depth = int(level.max())
        for k in range(depth):
            m = lu == k
            sigma += _gather_add(V, w[m], sigma[u[m]])
        dep = torch.zeros(V, dtype=torch.float64, device="cuda")
        for k in range(depth - 1, -1, -1):
            m = lu == k
            dep += sigma * _gather_add(V, u[m], (1.0 + dep[w[m]]) / sigma[w[m]])
        dep[s] = 0.0
        score += dep
    return score


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "ppr":
        return _exact_ppr(x)
    if kind == "bfs":
        return [_exact_levels(x, s) for s in x["sources"]]
    if kind == "bc":
        return _exact_bc(x)
    if kind == "spmv":
        src, _ = _rows(x["rowptr"])
        return _gather_add(x["V"], src, x["vals"].double() * x["x"].double()[x["colidx"].long()])
    r = _exact_pagerank(x)
    return r.cpu() if kind == "job" else r
