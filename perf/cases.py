"""The work that users of the library have it do, as measurable cases.

A case names a kind of call (one search, many searches into host memory, a
batch plan, a multi-source batch, a burst of served queries), the graph family
it runs on and the sizes.  Graphs are drawn on the GPU with torch from the seed
alone; sources are vertices with at least one entry in their column.  The
families are those of the repository's own workloads: Erdos-Renyi and R-MAT
(low diameter), a 4-neighbour grid and a directed 4-nearest-neighbour geometric
graph (large diameter).
"""
import math

import torch

import paper_1906_03113_gb300 as abfs

# quadrant probabilities of the R-MAT graphs
_A, _B, _C = 0.57, 0.19, 0.19


def listed():
    return [
        # the smallest call: a query on a neighbourhood-sized graph, where the
        # launches and the latency of a level are everything
        dict(name="run_er_1k", kind="run", graph="er", n=1000, degree=8.0),
        # one search on a mid-sized sparse graph that stays in cache
        dict(name="run_er_64k", kind="run", graph="er", n=65536, degree=8.0),
        # the headline: one search on a large social-network-like graph
        dict(name="run_rmat22", kind="run", graph="rmat", scale=22, edge_factor=16.0),
        # the same family after abfs_graph_relabel, which a program that keeps
        # a skewed graph resident calls once
        dict(name="relabel_rmat20", kind="relabel", graph="rmat", scale=20, edge_factor=16.0),
        # direction-optimising searches (bottom_up_alpha), the fastest option on
        # skewed graphs
        dict(name="hybrid_rmat21", kind="hybrid", graph="rmat", scale=21, edge_factor=16.0),
        # shortest-path counts, as betweenness-style programs need them
        dict(name="counts_rmat20", kind="counts", graph="rmat", scale=20, edge_factor=16.0),
        # road-network-like: thousands of thin levels
        dict(name="run_grid_4096", kind="run", graph="grid", width=4096, height=4096),
        # road-network-like, directed and irregular
        dict(name="run_rgg_4m", kind="run", graph="rgg", n=1 << 22),
        # many independent graphs of uneven size as one plan, launched again
        # and again (degrees of 4..32, sizes over a factor of 256)
        dict(name="batch_128", kind="batch", count=128, lo=10.0, hi=18.0),
        # 64 searches on one large graph as one plan (landmark distances)
        dict(name="multi64_rmat22", kind="multi", graph="rmat", scale=22, edge_factor=16.0,
             sources=64),
        # a burst of queries on resident graphs of mixed sizes through the server
        dict(name="serve_burst", kind="serve", queries=256, lo=12.0, hi=19.0, graphs=16),
        # searches whose results go to pinned host memory
        dict(name="host_rmat20", kind="host", graph="rmat", scale=20, edge_factor=16.0, sources=8),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "relabel", "hybrid", "counts", "batch", "multi",
                       "serve", "host"])
    if kind == "batch":
        lo = rng.uniform(10.0, 14.0)
        return dict(kind=kind, count=rng.randint(8, 128), lo=lo, hi=rng.uniform(lo, 18.0))
    if kind == "serve":
        lo = rng.uniform(10.0, 14.0)
        return dict(kind=kind, queries=rng.randint(32, 256), lo=lo, hi=rng.uniform(lo, 19.0),
                    graphs=rng.randint(2, 16))
    families = {"run": ["er", "rmat", "grid", "rgg"], "relabel": ["rmat"], "hybrid": ["er", "rmat"],
                "counts": ["er", "rmat", "grid"], "multi": ["er", "rmat"], "host": ["er", "rmat"]}
    c = dict(kind=kind, graph=rng.choice(families[kind]))
    if c["graph"] == "er":
        c["n"] = _log_uniform(rng, 500, 1 << 20)
        c["degree"] = rng.uniform(3.0, 24.0)
    elif c["graph"] == "rmat":
        c["scale"] = rng.randint(12, 20 if kind in ("relabel", "multi", "host") else 22)
        c["edge_factor"] = rng.uniform(4.0, 16.0)
    elif c["graph"] == "grid":
        c["width"] = _log_uniform(rng, 30, 4096)
        c["height"] = _log_uniform(rng, 30, 4096)
    else:
        c["n"] = _log_uniform(rng, 2000, 1 << 22)
    if kind == "multi":
        c["sources"] = rng.randint(8, 64)
    elif kind == "host":
        c["sources"] = rng.randint(1, 12)
    return c


# ---------------------------------------------------------------------------
# graphs: (colptr int64[n+1], rowidx int64[nnz], directed) on the GPU
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _csc(n, cols, rows):
    """CSC of the distinct pairs (column, row), rows ascending in each column."""
    key = torch.unique(cols * n + rows)
    cols = torch.div(key, n, rounding_mode="floor")
    rows = key - cols * n
    colptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    colptr[1:] = torch.cumsum(torch.bincount(cols, minlength=n), 0)
    return colptr, rows


def _undirected(n, a, b):
    keep = a != b
    a, b = a[keep], b[keep]
    return _csc(n, torch.cat([a, b]), torch.cat([b, a]))


def _er(n, degree, seed):
    g = _gen(seed)
    m = int(n * degree / 2)
    a = torch.randint(0, n, (m,), generator=g, device="cuda")
    b = torch.randint(0, n, (m,), generator=g, device="cuda")
    return _undirected(n, a, b) + (False,)


def _rmat(n, scale, edge_factor, seed):
    """R-MAT with labels randomly permuted, truncated to the first n labels."""
    g = _gen(seed)
    m = int((1 << scale) * edge_factor)
    a = torch.zeros(m, dtype=torch.int64, device="cuda")
    b = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        u = torch.rand(m, generator=g, device="cuda")
        ra = u >= _A + _B
        rb = ((u >= _A) & (u < _A + _B)) | (u >= _A + _B + _C)
        a = 2 * a + ra
        b = 2 * b + rb
    perm = torch.randperm(1 << scale, generator=g, device="cuda")
    a, b = perm[a], perm[b]
    keep = (a < n) & (b < n)
    return _undirected(n, a[keep], b[keep]) + (False,)


def _grid(width, height):
    n = width * height
    v = torch.arange(n, device="cuda")
    c, r = v % width, torch.div(v, width, rounding_mode="floor")
    # neighbours in ascending order: up, left, right, down
    cand = torch.stack([v - width, v - 1, v + 1, v + width], 1)
    ok = torch.stack([r > 0, c > 0, c < width - 1, r < height - 1], 1)
    colptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    colptr[1:] = torch.cumsum(ok.sum(1), 0)
    return colptr, cand[ok], False


def _rgg(n, seed, k=4, cap=12):
    """Arcs from each of n uniform points to its k nearest among the points of
    the 3 x 3 cells around it (about three points per cell)."""
    g = _gen(seed)
    side = max(1, int(math.sqrt(n / 3.0)))
    xy = torch.rand(n, 2, generator=g, device="cuda")
    cell = (xy * side).long().clamp_(max=side - 1)
    cid = cell[:, 1] * side + cell[:, 0]
    order = torch.argsort(cid, stable=True)
    start = torch.zeros(side * side + 1, dtype=torch.int64, device="cuda")
    start[1:] = torch.cumsum(torch.bincount(cid, minlength=side * side), 0)
    slots = torch.arange(cap, device="cuda")
    cols, rows = [], []
    for lo in range(0, n, 1 << 19):
        v = torch.arange(lo, min(n, lo + (1 << 19)), device="cuda")
        cand = []
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                x, y = cell[v, 0] + dx, cell[v, 1] + dy
                inside = (x >= 0) & (x < side) & (y >= 0) & (y < side)
                c = torch.where(inside, y * side + x, 0)
                at = start[c][:, None] + slots
                good = inside[:, None] & (at < start[c + 1][:, None])
                cand.append(torch.where(good, order[at.clamp(max=n - 1)], -1))
        cand = torch.cat(cand, 1)
        d = (xy[cand.clamp(min=0)] - xy[v][:, None]).square().sum(2)
        d[(cand < 0) | (cand == v[:, None])] = 9.0
        best, at = torch.topk(d, k, dim=1, largest=False)
        near = torch.gather(cand, 1, at)
        keep = best < 9.0
        cols.append(v[:, None].expand(-1, k)[keep])
        rows.append(near[keep])
    return _csc(n, torch.cat(cols), torch.cat(rows)) + (True,)


def _build(case, seed):
    if case["graph"] == "er":
        return _er(case["n"], case["degree"], seed)
    if case["graph"] == "rmat":
        return _rmat(1 << case["scale"], case["scale"], case["edge_factor"], seed)
    if case["graph"] == "grid":
        return _grid(case["width"], case["height"])
    return _rgg(case["n"], seed)


def _many(count, lo, hi, seed):
    """count ER and R-MAT graphs in turn, n spread log-uniformly over [2^lo, 2^hi]
    and the degree over 4..32 (the sizes are the case's, the edges the seed's)."""
    out = []
    for i in range(count):
        a, b = (0.6180339887 * i + 0.37) % 1.0, (0.7548776662 * i + 0.11) % 1.0
        n, d = int(round(2.0 ** (lo + (hi - lo) * a))), 4.0 + 28.0 * b
        if i % 2 == 0:
            out.append(_er(n, d, seed * 1009 + i))
        else:
            out.append(_rmat(n, max(1, math.ceil(math.log2(n))), d / 2, seed * 1009 + i))
    return out


def _sources(colptr, count, seed):
    """count distinct vertices with a non-empty column (all of them if fewer)."""
    cand = torch.nonzero(colptr[1:] > colptr[:-1]).flatten()
    at = torch.randperm(cand.numel(), generator=_gen(seed + 7), device="cuda")
    return cand[at[:count]].tolist()


def _queries(case, seed):
    """The graphs of a serving case and its (graph, source) queries."""
    graphs = _many(case["graphs"], case["lo"], case["hi"], seed)
    srcs = [_sources(g[0], case["queries"], seed + i) for i, g in enumerate(graphs)]
    which = [int(len(graphs) * ((0.5698402910 * q + 0.23) % 1.0)) for q in range(case["queries"])]
    return graphs, [(g, srcs[g][q % len(srcs[g])]) for q, g in enumerate(which)]


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _handle(g):
    colptr, rowidx, directed = g
    return abfs.graph_create(colptr.to(torch.int32), rowidx.to(torch.int32), directed=directed)


def _outputs(sizes):
    """One level and one parent buffer, and each query's views into them (every
    view starts on 16 elements)."""
    at, total = [], 0
    for n in sizes:
        at.append(total)
        total += (n + 15) // 16 * 16
    level = torch.full((total,), -2, dtype=torch.int32, device="cuda")
    parent = torch.full((total,), -2, dtype=torch.int32, device="cuda")
    return (level, parent, [level[a:a + n] for a, n in zip(at, sizes)],
            [parent[a:a + n] for a, n in zip(at, sizes)])


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "batch":
        graphs = _many(case["count"], case["lo"], case["hi"], seed)
        srcs = [_sources(g[0], 1, seed)[0] for g in graphs]
        st["graphs"] = [_handle(g) for g in graphs]
        st["level"], st["parent"], lv, pr = _outputs([g.n for g in st["graphs"]])
        st["plan"] = abfs.BatchPlan(st["graphs"], srcs, levels=lv, parents=pr)
        return st
    if kind == "serve":
        graphs, st["queries"] = _queries(case, seed)
        st["graphs"] = [_handle(g) for g in graphs]
        st["level"], st["parent"], st["lv"], st["pr"] = _outputs(
            [st["graphs"][g].n for g, _ in st["queries"]])
        # a program that also uses the GPU for other work lets the server's
        # launch end soon after its queue has emptied
        cfg = abfs.serve_default_cfg(max_slots=128, memory_budget=2 << 30, idle_exit_ms=2)
        st["server"] = abfs.Server(st["graphs"], cfg)
        return st
    g = _build(case, seed)
    st["srcs"] = _sources(g[0], case.get("sources", 1), seed)
    G = st["graph"] = _handle(g)
    if kind == "relabel":
        abfs.graph_relabel(G)
    elif kind == "hybrid":
        st["params"] = abfs.default_params(bottom_up_alpha=5)
    elif kind == "multi":
        srcs = st["srcs"]
        st["level"], st["parent"], lv, pr = _outputs([G.n] * len(srcs))
        st["plan"] = abfs.BatchPlan([G] * len(srcs), srcs, levels=lv, parents=pr)
    elif kind == "host":
        shape = (len(st["srcs"]), G.n)
        st["level"] = torch.empty(shape, dtype=torch.int32).pin_memory()
        st["parent"] = torch.empty(shape, dtype=torch.int32).pin_memory()
    return st


def run(state):
    kind = state["kind"]
    if kind in ("run", "relabel"):
        return abfs.run(state["graph"], state["srcs"][0])
    if kind == "hybrid":
        return abfs.run(state["graph"], state["srcs"][0], params=state["params"])
    if kind == "counts":
        return abfs.run_counts(state["graph"], state["srcs"][0])
    if kind in ("batch", "multi"):
        state["plan"].launch()
        return state["level"], state["parent"]
    if kind == "host":
        level, parent, status = abfs.run_host_many(state["graph"], state["srcs"], state["level"],
                                                   state["parent"])
        return level, parent, max(status)
    server = state["server"]
    tickets = [server.submit(g, s, state["lv"][q], state["pr"][q])
               for q, (g, s) in enumerate(state["queries"])]
    status = [server.wait(t) for t in tickets]
    return state["level"], state["parent"], max(status)


# expected stored entries of the graph families
def _nnz(case):
    if case["graph"] == "er":
        return case["n"] * case["degree"]
    if case["graph"] == "rmat":
        return 2.0 * case["edge_factor"] * (1 << case["scale"]) * 0.95
    if case["graph"] == "grid":
        return 4.0 * case["width"] * case["height"]
    return 4.0 * case["n"]


def _n(case):
    if case["graph"] == "rmat":
        return 1 << case["scale"]
    return case["width"] * case["height"] if case["graph"] == "grid" else case["n"]


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        # mean of 2^U[lo, hi]; degree 18 on average
        span = max(case["hi"] - case["lo"], 1e-6) * math.log(2.0)
        n = (2.0 ** case["hi"] - 2.0 ** case["lo"]) / span if span > 1e-3 else 2.0 ** case["lo"]
        graphs = case["count"] if kind == "batch" else case["graphs"]
        searches = graphs if kind == "batch" else case["queries"]
        return {"bytes": graphs * n * 4.0 * 19 + searches * n * 8.0, "flops": searches * n * 18.0}
    n, nnz = float(_n(case)), _nnz(case)
    searches = case.get("sources", 1)
    out = 16.0 if kind == "counts" else 8.0
    # the matrix read once; level and parent (and counts) written once per
    # search; one semiring product per stored entry and search
    return {"bytes": 4.0 * (n + 1) + 4.0 * nnz + searches * out * n, "flops": searches * nnz}


# ---------------------------------------------------------------------------
# exact results: a frontier-by-frontier search in 64-bit torch
# ---------------------------------------------------------------------------

def _search(colptr, rowidx, src, counts=False):
    n = colptr.numel() - 1
    level = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    parent = torch.full((n,), n, dtype=torch.int64, device="cuda")
    tag = torch.empty(n, dtype=torch.int64, device="cuda")
    sigma = torch.zeros(n, dtype=torch.int64, device="cuda")
    f = torch.tensor([src], device="cuda")
    level[src], parent[src], sigma[src], k = 0, src, 1, 0
    while f.numel():
        beg = colptr[f]
        ln = colptr[f + 1] - beg
        first = torch.cumsum(ln, 0) - ln
        j = torch.repeat_interleave(f, ln)
        at = torch.arange(j.numel(), device="cuda") + torch.repeat_interleave(beg - first, ln)
        r = rowidx[at]
        new = level[r] < 0
        r, j = r[new], j[new]
        parent.scatter_reduce_(0, r, j, "amin")
        if counts:
            sigma.index_add_(0, r, sigma[j])
        x = torch.arange(r.numel(), device="cuda")
        tag[r] = x
        f = r[tag[r] == x]
        k += 1
        level[f] = k
    parent[level < 0] = -1
    return level.to(torch.int32), parent.to(torch.int32), sigma


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        if kind == "batch":
            graphs = _many(case["count"], case["lo"], case["hi"], seed)
            queries = [(i, _sources(g[0], 1, seed)[0]) for i, g in enumerate(graphs)]
        else:
            graphs, queries = _queries(case, seed)
        level, parent, lv, pr = _outputs([graphs[g][0].numel() - 1 for g, _ in queries])
        for q, (g, s) in enumerate(queries):
            a, b, _ = _search(graphs[g][0], graphs[g][1], s)
            lv[q].copy_(a)
            pr[q].copy_(b)
        return (level, parent) if kind == "batch" else (level, parent, 0)
    colptr, rowidx, _ = _build(case, seed)
    srcs = _sources(colptr, case.get("sources", 1), seed)
    if kind == "multi":
        n = colptr.numel() - 1
        level, parent, lv, pr = _outputs([n] * len(srcs))
        for q, s in enumerate(srcs):
            a, b, _ = _search(colptr, rowidx, s)
            lv[q].copy_(a)
            pr[q].copy_(b)
        return level, parent
    if kind == "host":
        got = [_search(colptr, rowidx, s) for s in srcs]
        return torch.stack([a for a, _, _ in got]), torch.stack([b for _, b, _ in got]), 0
    level, parent, sigma = _search(colptr, rowidx, srcs[0], kind == "counts")
    return (level, parent, sigma) if kind == "counts" else (level, parent)
