"""Servers on the level-synchronous engine: which CTAs stay, and which servers
run on it."""
import time

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


def _outputs(n):
    return [torch.full((n,), 7, dtype=torch.int32, device="cuda") for _ in range(2)]


def _exact(lev, par, want):
    return np.array_equal(lev.cpu().numpy(), want[0]) and np.array_equal(par.cpu().numpy(), want[1])


def test_ctas_without_work_stay_while_a_search_runs():
    """idle_exit_ms runs out many times over during a deep search on a part of
    the GPU; queries that come meanwhile are answered at once, by CTAs that were
    idle, and long before the deep search ends."""
    n = 400000
    path = synth.from_arcs(n, list(range(n - 1)), list(range(1, n)), directed=True)
    small = synth.er(20000, 8.0, seed=3)
    P, E = (abfs.graph_create(g.colptr, g.rowidx, directed=g.directed) for g in (path, small))
    want = [oracle.bfs(small, s) for s in range(8)]
    srv = abfs.Server([P, E], abfs.serve_default_cfg(max_slots=16, memory_budget=1 << 30, idle_exit_ms=1))
    outs = [_outputs(path.n)] + [_outputs(small.n) for _ in range(8)]
    torch.cuda.synchronize()
    # (the first launch of the process loads the kernel)
    assert srv.wait(srv.submit(1, 0, *outs[1])) == 0
    deep = srv.submit(0, 0, *outs[0])
    time.sleep(0.03)
    tickets = [srv.submit(1, s, *outs[1 + s]) for s in range(8)]
    assert [srv.wait(t) for t in tickets] == [0] * 8
    done_early = srv.poll(deep)[0]
    assert srv.wait(deep) == 0
    assert not done_early
    rep = srv.stop()
    assert rep["completed"] == 10 and rep["failed"] == 0
    assert torch.equal(outs[0][0], torch.arange(n, dtype=torch.int32, device="cuda"))
    for s in range(8):
        assert _exact(*outs[1 + s], want[s]), s
    for G in (P, E):
        G.destroy()


def test_bursts_around_the_idle_exit():
    """Single queries and bursts at gaps around idle_exit_ms: whether a query
    meets the launch or finds it ending, it is answered."""
    g = synth.rmat(14, 8.0, seed=3)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    srcs = [int(x) for x in synth.sources_with_degree(g, 6, seed=5)]
    want = [oracle.bfs(g, s) for s in srcs]
    srv = abfs.Server([G], abfs.serve_default_cfg(max_slots=4, memory_budget=1 << 28, idle_exit_ms=1))
    outs = [_outputs(g.n) for _ in srcs]
    rng = np.random.default_rng(9)
    count = 0
    for _ in range(120):
        time.sleep(float(rng.uniform(0.0007, 0.0016)))
        k = int(rng.integers(1, 7))
        tickets = [srv.submit(0, srcs[q], *outs[q]) for q in range(k)]
        assert [srv.wait(t) for t in tickets] == [0] * k
        count += k
    torch.cuda.synchronize()
    for q, w in enumerate(want):
        assert _exact(*outs[q], w), q
    rep = srv.stop()
    assert rep["completed"] == count and rep["failed"] == 0 and rep["launches"] > 1
    G.destroy()


@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 1])
def test_servers_on_either_side_of_the_team_limit(n):
    """The largest graph that is served by teams, and the smallest beside which
    every query goes to the unit scheduler: the same answers, for the small
    graph's queries too."""
    big, small = synth.er(n, 6.0, seed=4), synth.rmat(12, 8.0, seed=4)
    dev = [abfs.graph_create(g.colptr, g.rowidx, directed=False) for g in (big, small)]
    src = [int(np.argmax(g.degrees())) for g in (big, small)]
    want = [oracle.bfs(g, s) for g, s in zip((big, small), src)]
    srv = abfs.Server(dev, abfs.serve_default_cfg(max_slots=8, memory_budget=1 << 30, idle_exit_ms=2))
    jobs = []
    for q in range(12):
        i = q % 3 != 0
        jobs.append((int(i), *_outputs((big, small)[i].n)))
    torch.cuda.synchronize()
    tickets = [srv.submit(i, src[i], lev, par) for i, lev, par in jobs]
    assert [srv.wait(t) for t in tickets] == [0] * 12
    for i, lev, par in jobs:
        assert _exact(lev, par, want[i])
    assert srv.stop()["failed"] == 0
    for G in dev:
        G.destroy()


def _burst_ms(dev, params, outs, src, reps=11):
    """The median time of a burst of one query per output pair."""
    cfg = abfs.serve_default_cfg(max_slots=32, memory_budget=1 << 30, idle_exit_ms=50)
    cfg.params = params
    srv = abfs.Server([dev], cfg)
    times = []
    for _ in range(reps):
        t0 = time.perf_counter()
        tickets = [srv.submit(0, src + q, *out) for q, out in enumerate(outs)]
        assert [srv.wait(t) for t in tickets] == [0] * len(outs)
        times.append((time.perf_counter() - t0) * 1e3)
    assert srv.stop()["failed"] == 0
    return sorted(times)[reps // 2]


def test_no_query_of_a_burst_is_left_to_one_cta():
    """Sixteen deep queries, more than the CTAs that come free at a time make up
    teams for: the burst takes no longer than on the unit scheduler (it took
    twice as long while a late CTA took the last query alone)."""
    m = 64
    v = np.arange(m ** 3)
    x, y, z = v % m, (v // m) % m, v // (m * m)
    a = np.concatenate([v[x < m - 1], v[y < m - 1], v[z < m - 1]])
    b = np.concatenate([v[x < m - 1] + 1, v[y < m - 1] + m, v[z < m - 1] + m * m])
    g = synth.from_arcs(m ** 3, a.tolist(), b.tolist(), directed=False)
    G = abfs.graph_create(g.colptr, g.rowidx, directed=False)
    src = int(g.n // 2 + m // 2)
    outs = [_outputs(g.n) for _ in range(16)]
    torch.cuda.synchronize()
    scheduler = abfs.default_params(cluster_edges=abfs.default_params().cluster_edges - 1)
    slow = _burst_ms(G, scheduler, outs, src)
    fast = _burst_ms(G, abfs.default_params(), outs, src)
    for q in (0, 15):
        assert _exact(*outs[q], oracle.bfs(g, src + q))
    assert fast < 1.3 * slow, (fast, slow)
    G.destroy()
