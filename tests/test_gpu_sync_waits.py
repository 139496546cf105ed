"""Waits of the level-synchronous engine that run out, and the state that its
CTAs share across levels and searches."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1906_03113_gb300 as abfs  # noqa: E402
from paper_1906_03113_gb300 import binding  # noqa: E402


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    abfs.build()
    torch.cuda.set_device(0)
    return abfs.load()


def _star(leaves):
    """A directed star on the device: vertex 0 reaches every other."""
    colptr = torch.full((leaves + 2,), leaves, dtype=torch.int32, device="cuda")
    colptr[0] = 0
    rowidx = torch.arange(1, leaves + 1, dtype=torch.int32, device="cuda")
    return abfs.graph_create(colptr, rowidx, directed=True)


def _hold_each_barrier(lib, search, exact, at_least, at_most=60):
    """Holds barrier 0, 1, ... of `search` until it has no more barriers: each
    held search times out, and the one after it is exact."""
    for b in range(at_most):
        assert lib.abfs_test_hold_barrier(1, b) == 0
        try:
            status = search()
        finally:
            assert lib.abfs_test_hold_barrier(0, 0) == 0
        torch.cuda.synchronize()
        if status == 0:
            assert exact() and b >= at_least
            return
        assert status == binding.ERR_TIMEOUT, (b, status)
        assert search() == 0 and exact(), b
    raise AssertionError("more barriers than expected")


CASES = {
    # (graph, barriers at least): hubs whose lists overflow and are evened out;
    # thin, wide and again thin levels; thin levels only
    "spill": (lambda: synth.from_arcs(9002, [0] * 9000 + list(range(1, 9001)),
                                      list(range(1, 9001)) + [9001] * 9000, directed=True), 3),
    "rmat": (lambda: synth.rmat(17, 16.0, seed=11), 6),
    "er": (lambda: synth.er(30000, 4.0, seed=7), 8),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("kind", ["plain", "relabel", "hybrid", "counts"])
def test_each_wait_of_a_search_times_out(lib, name, kind):
    make, at_least = CASES[name]
    g = make()
    G = abfs.graph_create(g.colptr, g.rowidx, directed=g.directed)
    if kind == "relabel":
        abfs.graph_relabel(G)
    s = int(np.argmax(g.degrees())) if name != "er" else 5
    lo, po = oracle.bfs(g, s)
    so = oracle.path_counts(g, s) if kind == "counts" else None
    p = abfs.default_params(timeout_ms=2, **({"bottom_up_alpha": 4} if kind == "hybrid" else {}))
    out = {}

    def search():
        try:
            if kind == "counts":
                out["l"], out["p"], out["s"], _ = abfs.run_counts(G, s, params=p, stats=True)
            else:
                out["l"], out["p"], _ = abfs.run(G, s, params=p, stats=True)
            return 0
        except abfs.AbfsError as e:
            return e.status

    def exact():
        return (np.array_equal(out["l"].cpu().numpy(), lo) and np.array_equal(out["p"].cpu().numpy(), po)
                and (so is None or np.array_equal(out["s"].cpu().numpy().view(np.uint64), so)))

    _hold_each_barrier(lib, search, exact, 1 if kind == "hybrid" else at_least)
    G.destroy()


def test_each_wait_of_a_search_from_a_very_long_column_times_out(lib):
    """A source column with more items than the lists of the whole GPU hold
    starts in the global list, behind a barrier of its own."""
    leaves = 240 * 1024 * 256
    G = _star(leaves)
    p = abfs.default_params(timeout_ms=2)
    lev = torch.empty(leaves + 1, dtype=torch.int32, device="cuda")
    par = torch.empty(leaves + 1, dtype=torch.int32, device="cuda")

    def search():
        lev.fill_(7)
        par.fill_(7)
        try:
            abfs.run(G, 0, lev, par, params=p, stats=True)
            return 0
        except abfs.AbfsError as e:
            return e.status

    def exact():
        return int(lev[0]) == 0 and bool((lev[1:] == 1).all()) and bool((par == 0).all())

    _hold_each_barrier(lib, search, exact, 4)
    G.destroy()


def test_each_wait_of_a_multi_source_search_times_out(lib):
    g = synth.rmat(13, 16.0, seed=3)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    srcs = [int(x) for x in synth.sources_with_degree(g, 16, seed=3)]
    want = [oracle.bfs(g, s) for s in srcs]
    p = abfs.default_params(timeout_ms=2)
    out = {}

    def search():
        out["l"], out["p"], st = abfs.run_batch([G] * 16, srcs, params=p)
        torch.cuda.synchronize()
        assert len(set(st)) == 1
        return st[0]

    def exact():
        return all(np.array_equal(a.cpu().numpy(), lo) and np.array_equal(b.cpu().numpy(), po)
                   for a, b, (lo, po) in zip(out["l"], out["p"], want))

    _hold_each_barrier(lib, search, exact, 4)
    G.destroy()


@pytest.mark.parametrize("layers,mids", [(400, 1500), (150, 5000), (3, 60000)])
def test_lists_that_overflow_right_after_a_slice(lib, layers, mids):
    """Layers of one hub, its `mids` rows and the next hub: the hub's rows
    overflow one CTA's list and are evened out through the global list, and the
    level after that, behind a thin level's barrier, the next hub's rows
    overflow into the same list again."""
    step = mids + 1
    hub = np.arange(layers, dtype=np.int64) * step
    mid = hub[:, None] + np.arange(1, step)
    src = np.concatenate([np.repeat(hub, mids), mid[:-1].ravel()])
    dst = np.concatenate([mid.ravel(), np.repeat(hub[1:], mids)])
    g = synth.from_arcs(layers * step, src.tolist(), dst.tolist(), directed=True)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=True)
    lo, po = oracle.bfs(g, 0)
    want = torch.from_numpy(lo).cuda(), torch.from_numpy(po).cuda()
    for rep in range(10):
        lev, par, st = abfs.run(G, 0, stats=True)
        assert torch.equal(lev, want[0]) and torch.equal(par, want[1]), rep
        assert st["reached"] == g.n and st["nnz_reached"] == g.nnz
    G.destroy()


def _deep_batch(n_deep, count, n_mid):
    """A path, whose search takes far longer than a batch plan (which knows
    vertices and entries only) expects, and `count` graphs of four entries per
    column but vertex 0's, which is empty: their teams are made up of CTAs that
    the path's search holds and of CTAs that are free at once."""
    path = synth.from_arcs(n_deep, list(range(n_deep - 1)), list(range(1, n_deep)), directed=True)
    rng = np.random.default_rng(n_mid)
    col = np.repeat(np.arange(1, n_mid), 4)
    row = rng.integers(n_mid, size=col.size)
    mid = synth.from_arcs(n_mid, col.tolist(), row.tolist(), directed=True)
    P, M = (abfs.graph_create(g.colptr, g.rowidx, directed=True) for g in (path, mid))
    return path, mid, P, M


@pytest.mark.parametrize("source", [0, 1])
def test_members_that_wait_for_a_search_elsewhere(lib, source):
    """A search whose members wait longer than timeout_ms for one that is still
    busy with a deep search never ends as done with outputs that were not
    written, whoever comes last."""
    path, mid, P, M = _deep_batch(100000, 90, 60000)
    lo, po = (torch.from_numpy(x).cuda() for x in oracle.bfs(mid, source))
    p = abfs.default_params(timeout_ms=2, multi_source=0)
    graphs = [P] + [M] * 90
    lv, pr = ([torch.full((G.n,), 7, dtype=torch.int32, device="cuda") for G in graphs] for _ in range(2))
    _, _, st = abfs.run_batch(graphs, [0] + [source] * 90, lv, pr, params=p)
    torch.cuda.synchronize()
    for q, s in enumerate(st):
        assert s in (0, binding.ERR_TIMEOUT)
        if s == 0 and q == 0:
            assert torch.equal(lv[0], torch.arange(P.n, dtype=torch.int32, device="cuda"))
        elif s == 0:
            assert torch.equal(lv[q], lo) and torch.equal(pr[q], po), q
    P.destroy()
    M.destroy()


def test_a_deep_search_is_progress_for_those_who_wait(lib):
    """timeout_ms bounds waits without progress: the members that wait for the
    deep search (a thousand times longer than timeout_ms planned for) find their
    own, and every search of the batch is exact."""
    path, mid, P, M = _deep_batch(100000, 90, 60000)
    lo, po = (torch.from_numpy(x).cuda() for x in oracle.bfs(mid, 1))
    p = abfs.default_params(timeout_ms=1, multi_source=0)
    lv, pr, st = abfs.run_batch([P] + [M] * 90, [0] + [1] * 90, params=p)
    torch.cuda.synchronize()
    assert st == [0] * 91
    k = torch.arange(P.n, dtype=torch.int32, device="cuda")
    assert torch.equal(lv[0], k) and torch.equal(pr[0], (k - 1).clamp_(min=0))
    for q in range(1, 91):
        assert torch.equal(lv[q], lo) and torch.equal(pr[q], po), q
    P.destroy()
    M.destroy()
