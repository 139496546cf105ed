"""Searches of the level-synchronous engine at sizes that its plans have to look
at: many more vertices than entries, levels larger than a team's lists."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1906_03113_gb300 as abfs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    abfs.build()
    abfs.load()
    torch.cuda.set_device(0)


def _scheduler(**kw):
    """Parameters that send a search to the unit scheduler."""
    return abfs.default_params(cluster_edges=abfs.default_params().cluster_edges - 1, **kw)


def _us(search, reps=5):
    """The fastest of a few calls, after one that is not counted."""
    search()
    best = float("inf")
    for _ in range(reps):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        search()
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) * 1e3)
    return best


def _spread(n, m, seed):
    """An undirected graph of about m entries among m / 4 of n vertices, the
    others isolated, and a source that has entries."""
    rng = np.random.default_rng(seed)
    sub = np.sort(rng.permutation(n)[:max(m // 4, 2)])
    a, b = (sub[rng.integers(sub.size, size=m // 2)] for _ in range(2))
    keep = a != b
    return synth.from_arcs(n, a[keep].tolist(), b[keep].tolist(), directed=False), int(a[keep][0])


@pytest.mark.parametrize("n,m", [(20000, 1000), (1 << 16, 16384), (1 << 20, 1000), (1 << 22, 16384),
                                 ((1 << 25) + 3, 1 << 17), ((1 << 25) + 3, 1 << 20)])
def test_many_more_vertices_than_entries(n, m):
    """Exact on either side of the rules, and not slower than the unit scheduler
    by more than its time differs between runs (a factor of two: one CTA for
    such a search took ten to a hundred times as long)."""
    g, s = _spread(n, m, 7)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    lo, po = oracle.bfs(g, s)
    lev, par = abfs.run(G, s)
    assert np.array_equal(lev.cpu().numpy(), lo) and np.array_equal(par.cpu().numpy(), po)
    p = _scheduler()
    assert _us(lambda: abfs.run(G, s, lev, par)) < 2 * _us(lambda: abfs.run(G, s, lev, par, params=p))
    lv, pr, st = abfs.run_batch([G, G], [s, 0])
    torch.cuda.synchronize()
    assert st == [0, 0] and torch.equal(lv[0], lev) and torch.equal(pr[0], par)
    assert int((lv[1] >= 0).sum()) == int((oracle.bfs(g, 0)[0] >= 0).sum())
    G.destroy()


def _mesh(x, y, z):
    """A 6-neighbour mesh on the device: CSC and, per vertex, its coordinates."""
    n = x * y * z
    step = torch.tensor([-x * y, -x, -1, 1, x, x * y], device="cuda")
    ln, rows = [], []
    for lo in range(0, n, 1 << 24):
        v = torch.arange(lo, min(n, lo + (1 << 24)), device="cuda")
        ix, iy, iz = v % x, (v // x) % y, v // (x * y)
        ok = torch.stack([iz > 0, iy > 0, ix > 0, ix < x - 1, iy < y - 1, iz < z - 1], 1)
        ln.append(ok.sum(1))
        rows.append((v[:, None] + step)[ok].to(torch.int32))
    colptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    colptr[1:] = torch.cumsum(torch.cat(ln), 0)
    return colptr.to(torch.int32), torch.cat(rows)


def test_levels_longer_than_the_lists_of_the_whole_gpu():
    """A mesh whose middle levels have more vertices than the lists of all CTAs
    hold: exact (a vertex's level is its distance along the axes, its parent the
    least neighbour one level down), and not slower than the unit scheduler."""
    x, y, z = 430, 420, 410
    colptr, rowidx = _mesh(x, y, z)
    G = abfs.graph_create(colptr, rowidx, directed=False)
    n, s = x * y * z, x * y * (z // 2) + x * (y // 2) + x // 2
    lev, par = abfs.run(G, s)
    step = torch.tensor([-x * y, -x, -1, 1, x, x * y], device="cuda")
    for lo in range(0, n, 1 << 24):
        v = torch.arange(lo, min(n, lo + (1 << 24)), device="cuda")
        d = [v // (x * y) - z // 2, (v // x) % y - y // 2, v % x - x // 2]
        want = sum(a.abs() for a in d)
        assert torch.equal(lev[v].long(), want)
        # one step towards the source along each axis; the least of those
        toward = torch.stack([v - torch.sign(a) * t for a, t in zip(d, (x * y, x, 1))], 1)
        toward = torch.where(torch.stack(d, 1) == 0, n, toward)
        want = toward.min(1).values
        want[v == s] = s
        assert torch.equal(par[v].long(), want)
    widest = int(torch.bincount(lev).max())
    assert widest > 160 * 1024
    p = _scheduler()
    assert _us(lambda: abfs.run(G, s, lev, par), 3) < 1.2 * _us(lambda: abfs.run(G, s, lev, par, params=p), 3)
    G.destroy()


SMALL_TEAMS = {
    "mesh": lambda: synth.from_arcs(*_mesh_arcs(30, 30, 30)),
    "mesh_flat": lambda: synth.from_arcs(*_mesh_arcs(120, 60, 3)),
    # the frontier grows from a list's length to several of them and, with
    # thousands of entries per CTA more, into wide levels
    "er": lambda: synth.er(16000, 3.0, seed=5),
    "er_dense": lambda: synth.er(30000, 9.0, seed=6),
    # columns of several items whose rows overflow the list at once
    "hubs": lambda: synth.rmat(13, 10.0, seed=8),
}


def _mesh_arcs(x, y, z):
    v = np.arange(x * y * z)
    ix, iy, iz = v % x, (v // x) % y, v // (x * y)
    a = np.concatenate([v[ix < x - 1], v[iy < y - 1], v[iz < z - 1]])
    b = np.concatenate([v[ix < x - 1] + 1, v[iy < y - 1] + x, v[iz < z - 1] + x * y])
    return x * y * z, a.tolist(), b.tolist(), False


@pytest.mark.parametrize("name", list(SMALL_TEAMS))
@pytest.mark.parametrize("kind", ["plain", "counts", "hybrid"])
@pytest.mark.parametrize("count", [40, 200])
def test_levels_longer_than_a_small_team_s_lists(name, kind, count):
    """A batch in which each search has a few CTAs, or one, and levels of more
    items than these hold."""
    g = SMALL_TEAMS[name]()
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    srcs = [int(s) for s in synth.sources_with_degree(g, 5, seed=2)]
    want = [[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in oracle.bfs(g, s)] for s in srcs]
    sig = [oracle.path_counts(g, s).view(np.int64) for s in srcs] if kind == "counts" else None
    p = abfs.default_params(multi_source=0, **({"bottom_up_alpha": 4} if kind == "hybrid" else {}))
    plan = abfs.BatchPlan([G] * count, [srcs[q % 5] for q in range(count)], params=p, counts=kind == "counts")
    for rep in range(2):
        plan.launch()
        assert plan.status() == [0] * count
        for q in range(count):
            assert torch.equal(plan.levels[q], want[q % 5][0]), (rep, q)
            assert torch.equal(plan.parents[q], want[q % 5][1]), (rep, q)
            if sig:
                assert np.array_equal(plan.sigmas[q].cpu().numpy(), sig[q % 5]), (rep, q)
    plan.destroy()
    G.destroy()
