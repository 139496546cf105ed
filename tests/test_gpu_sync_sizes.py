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
