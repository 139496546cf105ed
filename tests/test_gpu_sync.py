"""The level-synchronous engine (default parameters) at the sizes where its
lists, items, bitmaps and vector loads change shape, against the oracle."""
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


def _hubs(lengths, seed):
    """A directed two-level tree: vertex 0 reaches one hub per length, hub i
    reaches that many leaves (shared among the hubs, so the least hub wins)."""
    leaves = max(lengths)
    first = 1 + len(lengths)
    src, dst = [], []
    rng = np.random.default_rng(seed)
    for i, m in enumerate(lengths):
        src.append(0)
        dst.append(1 + i)
        pick = rng.permutation(leaves)[:m] + first
        src.extend([1 + i] * m)
        dst.extend(pick.tolist())
    return synth.from_arcs(first + leaves, src, dst, directed=True)


GRAPHS = {
    # column lengths around an item (256 entries less the head) and two, at
    # every alignment of the column's start
    "items": lambda: _hubs([1, 2, 3, 4, 5, 253, 254, 255, 256, 257, 258, 259, 509, 511, 512, 513, 1027], 1),
    # one CTA's list overflows into the global list, then is evened out
    "spill": lambda: _hubs([1500, 9000, 3000] + [2] * 3000, 2),
    "star": lambda: synth.from_arcs(300001, [0] * 300000, list(range(1, 300001)), directed=False),
    # dense enough for wide levels, from thin ones and back
    "wide": lambda: synth.rmat(17, 16.0, seed=11),
    "wide_er": lambda: synth.er(131071, 32.0, seed=12),
    # vertex counts off every vector width
    "odd": lambda: synth.rmat(13, 12.0, seed=13, n_keep=8190 - 27),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("shift", [0, 1])
def test_default_engine_at_its_edges(name, shift):
    g = GRAPHS[name]()
    G = abfs.graph_create(g.colptr, g.rowidx, directed=g.directed)
    deg = g.degrees()
    for relabel in (False, True):
        if relabel:
            abfs.graph_relabel(G)
        for s in sorted({0, int(np.argmax(deg)), g.n - 1}):
            # outputs off 16-byte alignment when shift is 1
            lev, par = (torch.full((g.n + 1,), 7, dtype=torch.int32, device="cuda")[shift:shift + g.n]
                        for _ in range(2))
            lo, po = oracle.bfs(g, s)
            for kw in ({}, {"bottom_up_alpha": 4}):
                _, _, st = abfs.run(G, s, lev, par, params=abfs.default_params(**kw), stats=True)
                assert np.array_equal(lev.cpu().numpy(), lo), (name, s, kw)
                assert np.array_equal(par.cpu().numpy(), po), (name, s, kw)
                assert st["reached"] == int((lo >= 0).sum()) and st["levels"] == int(lo.max()) + 1
                assert st["nnz_reached"] == int(deg[lo >= 0].sum())
    lev, par, sig, st = abfs.run_counts(G, s, stats=True)
    assert np.array_equal(sig.cpu().numpy().view(np.uint64), oracle.path_counts(g, s)), name
    assert st["entries_read"] == st["nnz_reached"]
    G.destroy()


def test_batch_teams_and_queue():
    """One launch in which large searches run on teams of several CTAs and small
    ones are taken from the queue, replayed; then the same with path counts."""
    hosts = [synth.rmat(17, 16.0, seed=21), synth.er(60000, 9.0, seed=22), synth.grid(70, 53),
             synth.from_arcs(1, [], [], directed=False), synth.rgg_knn(5000, 4, seed=23),
             synth.rmat(15, 8.0, seed=24)] + [synth.er(900 + 31 * i, 5.0, seed=30 + i) for i in range(200)]
    dev = [abfs.graph_create(g.colptr, g.rowidx, directed=g.directed) for g in hosts]
    srcs = [int(np.argmax(g.degrees())) if g.nnz else 0 for g in hosts]
    want = [oracle.bfs(g, s) for g, s in zip(hosts, srcs)]
    plan = abfs.BatchPlan(dev, srcs)
    for rep in range(3):
        for t in plan.levels + plan.parents:
            t.fill_(9)
        plan.launch()
        assert plan.status() == [0] * len(dev)
        for i, (lo, po) in enumerate(want):
            assert np.array_equal(plan.levels[i].cpu().numpy(), lo), (rep, i)
            assert np.array_equal(plan.parents[i].cpu().numpy(), po), (rep, i)
    plan.destroy()
    plan = abfs.BatchPlan(dev[:12], srcs[:12], counts=True)
    plan.launch()
    assert plan.status() == [0] * 12
    for i in range(12):
        assert np.array_equal(plan.levels[i].cpu().numpy(), want[i][0])
        assert np.array_equal(plan.sigmas[i].cpu().numpy().view(np.uint64), oracle.path_counts(hosts[i], srcs[i]))
    plan.destroy()
    for G in dev:
        G.destroy()


@pytest.mark.parametrize("leaves,count", [(2047, 5), (2049, 64), (9000, 63), (20000, 64)])
def test_multi_source_long_columns(leaves, count):
    """A hub whose column is scanned by a whole CTA: sources are leaves on both
    sides of the lane, warp and round boundaries of that scan (their bits reach
    the hub from exactly one entry each), and the other way round."""
    g = synth.from_arcs(leaves + 1, [0] * leaves, list(range(1, leaves + 1)), directed=False)
    edge = [1, 16, 17, 32, 33, 128, 129, 144, 145, 2047, 4096, 4097, 4112, 4113, 8192, 8193, leaves]
    srcs = [s for s in edge if s <= leaves][:count - 1]
    rng = np.random.default_rng(leaves)
    srcs += [int(x) for x in rng.integers(leaves + 1, size=count - len(srcs))]
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    levels, parents, st = abfs.run_batch([G] * count, srcs)
    torch.cuda.synchronize()
    assert all(x == 0 for x in st)
    for s, L, P in zip(srcs, levels, parents):
        lo, po = oracle.bfs(g, s)
        assert np.array_equal(L.cpu().numpy(), lo) and np.array_equal(P.cpu().numpy(), po), s
    G.destroy()


def test_multi_source_on_a_skewed_graph():
    """64 sources on a graph with hubs and thousands of unreached vertices:
    pushed and pulled levels."""
    g = synth.rmat(16, 16.0, seed=31)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    srcs = [int(x) for x in synth.sources_with_degree(g, 64, seed=3)]
    levels, parents, st = abfs.run_batch([G] * 64, srcs)
    torch.cuda.synchronize()
    assert all(x == 0 for x in st)
    for s, L, P in zip(srcs, levels, parents):
        lo, po = oracle.bfs(g, s)
        assert np.array_equal(L.cpu().numpy(), lo) and np.array_equal(P.cpu().numpy(), po), s
    G.destroy()


@pytest.mark.parametrize("slots", [1, 3, 40])
def test_serving_teams(slots):
    """Queries large enough for teams of CTAs beside small ones, few slots (each
    reused) and many, two bursts with the device launch ended in between."""
    import time
    hosts = [synth.rmat(17, 16.0, seed=41), synth.er(20000, 10.0, seed=42), synth.er(700, 5.0, seed=43),
             synth.grid(60, 41)]
    dev = [abfs.graph_create(g.colptr, g.rowidx, directed=g.directed) for g in hosts]
    srcs = [synth.sources_with_degree(g, 8, seed=5) for g in hosts]
    want = {}
    srv = abfs.Server(dev, abfs.serve_default_cfg(max_slots=slots, memory_budget=1 << 30, idle_exit_ms=1))
    for burst in range(2):
        jobs = []
        for i in range(48):
            gi = i % len(hosts)
            s = int(srcs[gi][(i // 4 + burst) % 8])
            lev, par = (torch.full((hosts[gi].n,), 7, dtype=torch.int32, device="cuda") for _ in range(2))
            jobs.append([gi, s, lev, par])
        # the fills are done before a query may write (the server has its own stream)
        torch.cuda.synchronize()
        for job in jobs:
            job.append(srv.submit(*job))
        for gi, s, lev, par, t in jobs:
            assert srv.wait(t) == 0
        for gi, s, lev, par, t in jobs:
            if (gi, s) not in want:
                want[gi, s] = oracle.bfs(hosts[gi], s)
            lo, po = want[gi, s]
            assert np.array_equal(lev.cpu().numpy(), lo) and np.array_equal(par.cpu().numpy(), po), (gi, s)
        time.sleep(0.05)
    rep = srv.stop()
    assert rep["completed"] == 96 and rep["failed"] == 0
    for G in dev:
        G.destroy()


def _path(n, extra, seed):
    """A path over all n vertices in a shuffled order (as many levels as
    vertices) with `extra` directed chords backwards along it."""
    rng = np.random.default_rng(seed)
    order = rng.permutation(n)
    a = rng.integers(1, n, size=extra)
    b = (a * rng.random(extra)).astype(np.int64)
    src = np.concatenate([order[:-1], order[a]])
    dst = np.concatenate([order[1:], order[b]])
    return order, synth.from_arcs(n, src.tolist(), dst.tolist(), directed=True)


# around the largest graph that one CTA holds whole (4096 vertices, 40960 entries)
@pytest.mark.parametrize("n,entries", [(1, 0), (2, 1), (33, 70), (1023, 9000), (4095, 40960), (4096, 40960),
                                       (4096, 40961), (4097, 40000), (1500, 41000)])
def test_searches_held_by_one_cta(n, entries):
    if n == 1:
        g, srcs = synth.from_arcs(1, [], [], directed=False), [0]
    elif n == 2:
        g, srcs = synth.from_arcs(2, [0], [1], directed=True), [0, 1]
    else:
        order, g = _path(n, 2 * entries, 51)
        while g.nnz > entries:  # duplicates merge: thin out to the exact count
            keep = np.sort(np.random.default_rng(52).permutation(g.nnz)[:entries])
            col = np.repeat(np.arange(n), g.degrees())[keep]
            g = synth.from_arcs(n, col.tolist(), np.asarray(g.rowidx)[keep].tolist(), directed=True)
        assert g.nnz == entries or entries > 40960 or n < 1024
        srcs = [int(order[0]), int(order[n // 2]), int(order[-1])]
    G = abfs.graph_create(g.colptr, g.rowidx, directed=g.directed)
    deg = g.degrees()
    chain = _path(n, 0, 53) if n > 2 else None
    for s in srcs:
        lo, po = oracle.bfs(g, s)
        lev, par, st = abfs.run(G, s, stats=True)
        assert np.array_equal(lev.cpu().numpy(), lo) and np.array_equal(par.cpu().numpy(), po), s
        assert st["reached"] == int((lo >= 0).sum()) and st["levels"] == int(lo.max()) + 1
        assert st["nnz_reached"] == int(deg[lo >= 0].sum()) == st["entries_read"]
    G.destroy()
    if chain:
        order, g = chain
        G = abfs.graph_create(g.colptr, g.rowidx, directed=True)
        lo, po = oracle.bfs(g, int(order[0]))
        levels, parents, status = abfs.run_batch([G, G], [int(order[0])] * 2)
        torch.cuda.synchronize()
        assert status == [0, 0] and int(lo.max()) == n - 1
        for lev, par in zip(levels, parents):
            assert np.array_equal(lev.cpu().numpy(), lo) and np.array_equal(par.cpu().numpy(), po)
        G.destroy()


@pytest.mark.parametrize("n", [196607, 196608, 196609])
def test_bitmap_in_shared_memory_at_its_limit(n):
    """Wide levels around the largest graph whose bitmap fits beside the lists,
    on a large team, on the small teams of a batch, and with path counts."""
    rng = np.random.default_rng(n)
    # two dense halves of the vertex range, bridged: rows on the first and last words
    src = rng.integers(n, size=6 * n)
    dst = np.concatenate([rng.integers(n, size=5 * n), n - 1 - rng.integers(64, size=n)])
    g = synth.from_arcs(n, src.tolist(), dst.tolist(), directed=False)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    lo, po = oracle.bfs(g, n - 1)
    lev, par = abfs.run(G, n - 1)
    assert np.array_equal(lev.cpu().numpy(), lo) and np.array_equal(par.cpu().numpy(), po)
    lev, par, sig = abfs.run_counts(G, n - 1)
    assert np.array_equal(lev.cpu().numpy(), lo) and np.array_equal(par.cpu().numpy(), po)
    assert np.array_equal(sig.cpu().numpy().view(np.uint64), oracle.path_counts(g, n - 1))
    levels, parents, status = abfs.run_batch([G] * 7, [n - 1] * 7)
    torch.cuda.synchronize()
    assert status == [0] * 7
    for lev, par in zip(levels, parents):
        assert np.array_equal(lev.cpu().numpy(), lo) and np.array_equal(par.cpu().numpy(), po)
    G.destroy()
