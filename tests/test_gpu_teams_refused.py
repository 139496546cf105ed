"""Searches that would run on teams of CTAs where teams cannot run."""
import time

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")

import paper_1906_03113_gb300 as abfs  # noqa: E402


@pytest.fixture(scope="module")
def lib():
    abfs.build()
    return abfs.load()


def test_refuse_control_needs_no_device(lib):
    assert lib.abfs_test_refuse_teams(1) == 0
    assert lib.abfs_test_refuse_teams(0) == 0


def _same(got, want):
    return all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(got, want))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1000, 30000])
@pytest.mark.parametrize("relabel", [False, True])
def test_launches_that_the_device_does_not_take(lib, n, relabel):
    """A launch of CTAs that start together is refused (fewer SMs usable than the
    device reports): every call runs on the unit scheduler instead."""
    g = synth.er(n, 7.0, seed=3)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    if relabel:
        abfs.graph_relabel(G)
    srcs = [int(s) for s in synth.sources_with_degree(g, 12, seed=2)]
    want = [oracle.bfs(g, s) for s in srcs]
    assert lib.abfs_test_refuse_teams(1) == 0
    try:
        assert _same(abfs.run(G, srcs[0]), want[0])
        assert _same(abfs.run(G, srcs[1], params=abfs.default_params(bottom_up_alpha=4)), want[1])
        lev, par, sig = abfs.run_counts(G, srcs[2])
        assert _same((lev, par), want[2])
        assert np.array_equal(sig.cpu().numpy().view(np.uint64), oracle.path_counts(g, srcs[2]))
        lev, par, st = abfs.run_host_many(G, srcs[:4])
        assert st == [0] * 4 and all(np.array_equal(np.asarray(lev[q]), want[q][0]) for q in range(4))
        for multi in (0, 8):
            plan = abfs.BatchPlan([G] * 12, srcs, params=abfs.default_params(multi_source=multi))
            for _ in range(2):
                plan.launch()
                assert plan.status() == [0] * 12
                assert all(_same((plan.levels[q], plan.parents[q]), want[q]) for q in range(12))
            plan.destroy()
    finally:
        assert lib.abfs_test_refuse_teams(0) == 0
    assert _same(abfs.run(G, srcs[0]), want[0])
    G.destroy()


@pytest.mark.gpu
def test_searches_beside_a_server_that_leaves_room(lib):
    """A server with ctas_per_sm 1 keeps half of every SM for as long as it runs;
    searches, and plans made before it, run in the other half instead of waiting
    until it idles out."""
    g = synth.rmat(15, 8.0, seed=3)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    srcs = [int(s) for s in synth.sources_with_degree(g, 3, seed=2)]
    want = [oracle.bfs(g, s) for s in srcs]
    before = abfs.BatchPlan([G] * 3, srcs)
    before.launch()
    assert before.status() == [0] * 3
    # (kernels are loaded at their first use, which waits for the device)
    for t in before.levels + before.parents:
        t.fill_(9)
    unit = abfs.default_params(ctas_per_sm=1)
    abfs.run(G, srcs[0])
    abfs.run(G, srcs[0], params=unit)
    plan = abfs.BatchPlan([G] * 3, srcs, params=unit)
    plan.launch()
    assert plan.status() == [0] * 3
    plan.destroy()
    cfg = abfs.serve_default_cfg(max_slots=4, memory_budget=1 << 28, idle_exit_ms=3000)
    cfg.params = abfs.default_params(ctas_per_sm=1)
    srv = abfs.Server([G], cfg)
    out = [torch.empty(g.n, dtype=torch.int32, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    assert srv.wait(srv.submit(0, srcs[1], *out)) == 0  # its launch is there now
    t0 = time.perf_counter()
    got = abfs.run(G, srcs[0])
    torch.cuda.current_stream().synchronize()
    for t in before.levels + before.parents:
        t.fill_(7)
    before.launch()
    torch.cuda.current_stream().synchronize()
    dt = time.perf_counter() - t0
    assert before.status() == [0] * 3
    assert _same(got, want[0])
    for q in range(3):
        assert _same((before.levels[q], before.parents[q]), want[q])
    assert srv.stop()["failed"] == 0
    assert dt < 1.5, dt
    # and on teams again without it
    assert _same(abfs.run(G, srcs[2]), want[2])
    before.destroy()
    G.destroy()


class _Limit:
    """An allocator hook over torch that refuses blocks of more than `low` and at
    most `high` bytes."""

    def __init__(self, low, high):
        import ctypes
        self.live, self.refused = {}, 0

        def alloc(nbytes, ctx):
            if low < nbytes <= high:
                self.refused += 1
                return None
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr()] = t
            return t.data_ptr()

        self.a = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)(alloc)
        self.f = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)(lambda p, ctx: self.live.__delitem__(p))
        self.ptr = [ctypes.cast(x, ctypes.c_void_p) for x in (self.a, self.f)]


@pytest.mark.gpu
def test_memory_that_holds_a_search_of_the_scheduler_only(lib):
    """On a dense graph a team's lists take more than the scheduler's arrays.
    Servers, searches and batches that fit with the scheduler's run there."""
    n = 1200
    a, b = np.nonzero(np.random.default_rng(4).random((n, n)) < 0.4)
    g = synth.from_arcs(n, a.tolist(), b.tolist(), directed=False)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    need = G.footprint()
    # (smaller granules: a little more than the scheduler's own layout)
    unit = G.footprint(abfs.default_params(unit_entries=512))
    assert unit + 256 < need
    want = [oracle.bfs(g, s) for s in range(3)]
    srv = abfs.Server([G], abfs.serve_default_cfg(max_slots=4, memory_budget=unit + 256, idle_exit_ms=1))
    outs = [[torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2)] for _ in want]
    torch.cuda.synchronize()
    tickets = [srv.submit(0, s, *outs[s]) for s in range(3)]
    assert [srv.wait(t) for t in tickets] == [0] * 3
    assert srv.stop()["failed"] == 0
    assert all(_same(outs[s], want[s]) for s in range(3))
    with pytest.raises(abfs.AbfsError) as ei:
        abfs.Server([G], abfs.serve_default_cfg(memory_budget=unit // 2))
    assert ei.value.status == abfs.binding.ERR_OOM
    G.destroy()
    hook = _Limit(unit, need + 256)
    assert lib.abfs_set_allocator(*hook.ptr, None) == 0
    try:
        G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
        assert hook.refused == 0
        assert _same(abfs.run(G, 0), want[0]) and hook.refused == 1
        assert _same(abfs.run(G, 1), want[1]) and hook.refused == 1
        plan = abfs.BatchPlan([G], [2])
        plan.launch()
        assert plan.status() == [0] and _same((plan.levels[0], plan.parents[0]), want[2])
        assert hook.refused == 2
        plan.destroy()
        G.destroy()
    finally:
        assert lib.abfs_set_allocator(None, None, None) == 0
    assert not hook.live
