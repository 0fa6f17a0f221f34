"""Edges of the kernels' work splits: the sizes at which a tile, a pool, a
segment or a launch rule begins and ends, each against the oracle or against
the form of the same call that takes the other path."""

import numpy as np
import pytest

import oracle
from pw_inputs import barabasi_albert, complete_graph, cycle_graph, er_cycle, query_seeds, uniform_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    from paper_2512_05460_gb300 import build

    build.build()
    from paper_2512_05460_gb300 import probewalk

    probewalk.lib()
    return probewalk


# n = 5, 16: the 12-round permutation; 17: the smallest 8-round one; 33: n just
# above 2^b / 2, where cycle-walks are longest; 65: odd, one zero node
GRAPHS = [lambda: complete_graph(5), lambda: cycle_graph(16), lambda: complete_graph(17), lambda: er_cycle(33, 0.2, 3),
          lambda: er_cycle(65, 0.1, 4)]


@pytest.mark.parametrize("graph_fn", GRAPHS)
def test_visit_pool_edges(pw, oracle_lib, graph_fn):
    """Per-visit walks in warp pools of 4 visits a side: walk lengths around the
    pool's, replica counts around a warp's, every U_p and visit against the oracle."""
    host = graph_fn()
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for L in (0, 1, 2, 3, 4, 7, 8):
            for R in (2, 31, 32, 33):
                params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=2, G=3, R=R, walk_mode=1)
                cfg = oracle.budget_cfg(mode=oracle.MODE_FIXED, B=2, G=3, R=R)
                dev = pw.pw_debug_query(g.handle, host.n, 0, 3, 0.3, L, 77 + L, params, q_cap=64, u_cap=4096,
                                        want_visits=True)
                orc = oracle.query(host, 0, 3, 0.3, L, 77 + L, cfg, want_q=True, want_u=True, want_visits=True)
                np.testing.assert_array_equal(dev["u"], orc["u"])
                np.testing.assert_array_equal(dev["visits"], orc["visits"])
                np.testing.assert_array_equal(dev["q"], orc["q"])
                assert dev["beta"] == orc["beta"]
                assert pw.pw_query(g.handle, 0, 3, 0.3, L, 77 + L, params) == orc["beta"]


@pytest.mark.parametrize("mode", ["pilot", "fixed", "adaptive"])
def test_plans_across_the_fused_launch(pw, oracle_lib, mode):
    """Up to 256 queries are planned and scanned in one launch, more in two; a
    batch of either kind gives each query, the invalid ones among them, what it
    gets in smaller batches."""
    host = er_cycle(200, 8 / 199, 0)
    budget = {"pilot": {}, "fixed": {"budget_mode": pw.PW_BUDGET_FIXED, "B": 2, "G": 3, "R": 5},
              "adaptive": {"budget_mode": pw.PW_BUDGET_ADAPTIVE}}[mode]
    params = pw.make_params(**budget)
    count = 1100  # more than one query per thread of the scan
    s, t = uniform_pairs(host.n, count, 7)
    seeds = query_seeds(count, 8)
    eps = np.full(count, 0.45)
    t[5], s[300] = s[5], -1
    eps[256] = 2.0
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        whole, st = pw.pw_query_batch(g.handle, s, t, eps, 9, seeds, params)
        assert st[300] == st[256] == pw.PW_ERR_ARG and np.count_nonzero(st) == 2 and whole[5] == 0.0
        for lo, hi in ((0, 1), (1, 33), (33, 289), (289, 546), (546, 1100)):
            part, pst = pw.pw_query_batch(g.handle, s[lo:hi], t[lo:hi], eps[lo:hi], 9, seeds[lo:hi], params)
            np.testing.assert_array_equal(part, whole[lo:hi])
            np.testing.assert_array_equal(pst, st[lo:hi])
    if mode == "pilot":
        want, _, _ = oracle.query_many(host, s[:4], t[:4], 0.45, 9, seeds[:4])
        np.testing.assert_array_equal(whole[:4], want)


@pytest.mark.parametrize("G", [1, 2, 5, 24, 129, 300])
def test_median_by_rank(pw, oracle_lib, G):
    """Even and odd block counts below and above the block's 128 threads."""
    host = barabasi_albert(400, 3, 5)
    params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=9, G=G, R=3)
    cfg = oracle.budget_cfg(mode=oracle.MODE_FIXED, B=9, G=G, R=3)
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for s, t in ((1, 2), (0, 399)):
            assert pw.pw_query(g.handle, s, t, 0.3, 6, 5, params) == oracle.query(host, s, t, 0.3, 6, 5, cfg)["beta"]


def _hub_graph(n, degrees):
    """A ring whose first nodes also link to `degrees` others."""
    from pw_inputs import from_edges

    u, v = [np.arange(n)], [(np.arange(n) + 1) % n]
    for i, d in enumerate(degrees):
        u.append(np.full(d, i))
        v.append((np.arange(d) * ((n - 40) // d) + 20 + i) % n)
    return from_edges(n, np.concatenate(u), np.concatenate(v), name="hubs", keep_lcc=False)


@pytest.mark.parametrize("count", [1, 4, 5, 8, 9, 16, 17, 33])
def test_series_column_widths(pw, count):
    """4, 8, 16 or 32 columns a pass, odd and even lengths (h takes two steps at
    a time), rows of one segment, of several and of more than 64: FP64's values
    to 1e-9, and each query's bits whatever it shares the pass with."""
    from oracle import exact

    host = _hub_graph(6000, [62, 63, 64, 130, 4500])
    s, t = uniform_pairs(host.n, count, 50 + count)
    s[0] = 4
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for L in (0, 1, 2, 7):
            got = pw.pw_series_batch(g.handle, s, t, L)
            want = exact.series_beta_many(host.row_ptr, host.col_idx, host.n, s, t, L)
            np.testing.assert_allclose(got, want, rtol=1e-9, atol=0)
            alone = [pw.pw_series_batch(g.handle, s[i : i + 1], t[i : i + 1], L)[0] for i in (0, count - 1)]
            np.testing.assert_array_equal(alone, got[[0, count - 1]])


@pytest.mark.parametrize("n", [5, 16, 17, 33, 255, 257, 1024, 1025, 4095, 4096, 4097])
def test_team_tables(pw, oracle_lib, n):
    """Table walks of small graphs by teams of one to eight warps: node counts
    around a word, a warp's batch of 256, the pilot's limit and the kernel's;
    probe counts that make teams of eight, of few and of one.  The per-visit
    kernel gives the same estimates, the oracle the single query's replicas."""
    host = complete_graph(n) if n < 17 else (cycle_graph(n) if n > 1025 else er_cycle(n, min(0.2, 8 / n), 3))
    s, t = np.array([0, 1, 2]), np.array([n - 1, 3, 4])
    seeds = query_seeds(3, n)
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for B, G, R, L in ((1, 3, 300, 5), (7, 150, 65, 3), (40, 200, 33, 2), (40, 200, 2, 0)):
            got = []
            for mode in (1, 2):
                params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=B, G=G, R=R, walk_mode=mode)
                beta, st = pw.pw_query_batch(g.handle, s, t, 0.3, L, seeds, params)
                assert np.all(st == 0)
                got.append(beta)
            np.testing.assert_array_equal(got[0], got[1])
        params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=1, G=2, R=70, walk_mode=2)
        dev = pw.pw_debug_query(g.handle, host.n, 0, n - 1, 0.3, 6, 9, params, q_cap=8, u_cap=256, want_visits=True)
        orc = oracle.query(host, 0, n - 1, 0.3, 6, 9, oracle.budget_cfg(mode=oracle.MODE_FIXED, B=1, G=2, R=70),
                           want_q=True, want_u=True, want_visits=True)
        np.testing.assert_array_equal(dev["u"], orc["u"])
        np.testing.assert_array_equal(dev["visits"], orc["visits"])
        b = oracle.budget(host, 0, n - 1, 0.3, 6, 9)
        assert pw.pw_budget(g.handle, 0, n - 1, 0.3, 6, 9) == {k: b[k] for k in "BGKR"}


def test_ranked_records(pw):
    """A power-law graph whose col_idx and node records exceed 64 MB: walks read
    packed ranks by degree, and give the fused layout's trajectories and estimates
    in both walk kernels and the server."""
    from pw_inputs import rmat_native

    host = rmat_native(18, 80, (0.57, 0.19, 0.19, 0.05), 6)
    assert 4 * host.nnz + 16 * host.n > 64 << 20 and host.n <= 1 << 21
    s, t = uniform_pairs(host.n, 5, 71)
    s[0] = int(np.argmax(np.diff(host.row_ptr)))
    seeds = query_seeds(5, 72)
    flags = pw.LOAD_NO_CONNECTIVITY
    with pw.Graph(host.row_ptr, host.col_idx, flags=flags) as g, \
            pw.Graph(host.row_ptr, host.col_idx, flags=flags | pw.LOAD_FUSED) as f:
        assert pw.pw_profile(g.handle, enable=False)["layout"] == 2
        want, _ = pw.pw_query_batch(f.handle, s, t, 0.3, 21, seeds)
        for mode in (0, 1, 2):
            got, st = pw.pw_query_batch(g.handle, s, t, 0.3, 21, seeds, pw.make_params(walk_mode=mode))
            assert np.all(st == 0)
            np.testing.assert_array_equal(got, want)
        params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=1, G=2, R=40, walk_mode=1)
        q = [pw.pw_debug_query(h.handle, host.n, int(s[0]), int(t[0]), 0.3, 21, 5, params, q_cap=8, u_cap=128,
                               want_visits=True) for h in (g, f)]
        np.testing.assert_array_equal(q[0]["u"], q[1]["u"])
        np.testing.assert_array_equal(q[0]["visits"], q[1]["visits"])
        srv = pw.pw_server_create(g.handle, None, 1 << 24)
        try:
            tickets = [pw.pw_server_submit(srv, int(s[i]), int(t[i]), 0.3, 21, int(seeds[i])) for i in range(5)]
            pw.pw_server_drain(srv, 60000)
            np.testing.assert_array_equal([pw.pw_server_poll(srv, x)[1] for x in tickets], want)
        finally:
            pw.pw_server_destroy(srv)


@pytest.mark.parametrize("K0,R0", [(1, 2), (5, 7), (64, 8), (64, 9), (63, 31), (64, 32), (400, 32)])
def test_pilot_forms(pw, oracle_lib, K0, R0):
    """The pilot by a block per probe (few probes) and by a warp per probe, with
    replica counts that leave some of the block's warps without any: the budget
    and the estimate of one query and of several against the oracle."""
    host = barabasi_albert(3000, 3, 5)
    params, cfg = pw.make_params(pilot_K0=K0, pilot_R0=R0), oracle.budget_cfg(K0=K0, R0=R0)
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for L in (0, 5):
            b = oracle.budget(host, 3, 2999, 0.4, L, 11, cfg)
            assert pw.pw_budget(g.handle, 3, 2999, 0.4, L, 11, params) == {k: b[k] for k in "BGKR"}
            want = oracle.query(host, 3, 2999, 0.4, L, 11, cfg)["beta"]
            assert pw.pw_query(g.handle, 3, 2999, 0.4, L, 11, params) == want
            many, _ = pw.pw_query_batch(g.handle, np.full(9, 3), np.full(9, 2999), 0.4, L,
                                        np.full(9, 11, np.uint64), params)
            np.testing.assert_array_equal(many, want)


@pytest.mark.parametrize("n", [5, 32, 33, 257, 2047, 2048, 2049])
def test_server_small_graph_jobs(pw, n):
    """A burst on a small graph: jobs of several tables side by side (up to 2048
    nodes), tapering to one as the queue drains, give the batch's estimates; so
    does a lone query, whose jobs are single."""
    host = barabasi_albert(n, 3, 8)
    s, t = uniform_pairs(n, 40, 91)
    seeds = query_seeds(40, 92)
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        want, st = pw.pw_query_batch(g.handle, s, t, 0.2, 40, seeds)
        assert np.all(st == 0)
        srv = pw.pw_server_create(g.handle, None, 1 << 26)
        try:
            tickets = [pw.pw_server_submit(srv, int(s[i]), int(t[i]), 0.2, 40, int(seeds[i])) for i in range(40)]
            pw.pw_server_drain(srv, 60000)
            np.testing.assert_array_equal([pw.pw_server_poll(srv, x)[1] for x in tickets], want)
            one = pw.pw_server_submit(srv, int(s[7]), int(t[7]), 0.2, 40, int(seeds[7]))
            pw.pw_server_drain(srv, 60000)
            assert pw.pw_server_poll(srv, one)[1] == want[7]
        finally:
            pw.pw_server_destroy(srv)


@pytest.mark.parametrize("graph_fn,eps", [(lambda: barabasi_albert(400, 5, 5), 0.3), (lambda: er_cycle(200, 8 / 199, 0), 0.8)])
def test_adaptive_stops_after_the_first_stage(pw, oracle_lib, graph_fn, eps):
    """ADAPTIVE queries whose stopping rule keeps the first stage's probes, and so
    run none in the second, return the first stage's estimate: alone, in a batch
    with queries that go on, as a replayed launch, and level by level."""
    host = graph_fn()
    params = pw.make_params(budget_mode=pw.PW_BUDGET_ADAPTIVE)
    cfg = oracle.budget_cfg(mode=oracle.MODE_ADAPTIVE)
    first = (int(np.ceil(0.5 / eps**2)) + 3) // 4
    count = 40
    s, t = uniform_pairs(host.n, count, 7)
    seeds = query_seeds(count, 8)
    t[3], s[4] = s[3], -1  # no work and an invalid query beside them
    ok = np.arange(count) != 4
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for L in (0, 1, 2):
            want, budgets, _ = oracle.query_many(host, s[ok], t[ok], eps, L, seeds[ok], cfg)
            stops = np.flatnonzero(ok)[(budgets[:, 0] == first) & (s != t)[ok]]
            assert 0 < stops.size < count - 2
            for _ in range(3):  # eager, captured, replayed
                beta, st = pw.pw_query_batch(g.handle, s, t, eps, L, seeds, params)
                np.testing.assert_array_equal(beta[ok], want)
                assert st[4] == pw.PW_ERR_ARG and np.all(st[ok] == 0) and np.isnan(beta[4])
            assert beta[3] == 0.0
            i = int(stops[0])
            one = oracle.query(host, int(s[i]), int(t[i]), eps, L, int(seeds[i]), cfg)["beta"]
            assert pw.pw_query(g.handle, int(s[i]), int(t[i]), eps, L, int(seeds[i]), params) == one
        beta, stop, st = pw.pw_query_stabilized(g.handle, s[ok], t[ok], eps, 8, seeds[ok], params)
        assert np.all(st == 0)
        for j, i in enumerate(np.flatnonzero(ok)):
            want, want_stop, _ = oracle.stabilized(host, int(s[i]), int(t[i]), eps, 8, int(seeds[i]), cfg)
            assert (beta[j], stop[j]) == (want, want_stop)


def test_tables_of_several_graphs(pw):
    """Graphs with probe tables of over 48 KB (the last with the kernel's own shared
    memory) and the same table kernel: using a smaller one leaves the larger one's
    launches as they were."""
    graphs = [cycle_graph(n) for n in (500_000, 420_000, 393_000)]  # 62.5, 52.5 and 48 KB
    seeds = query_seeds(3, 5)
    with pw.Graph(graphs[0].row_ptr, graphs[0].col_idx) as a, \
            pw.Graph(graphs[1].row_ptr, graphs[1].col_idx) as b, pw.Graph(graphs[2].row_ptr, graphs[2].col_idx) as c:
        for count in (1, 2, 3):  # a new count: launched, not replayed
            s, t = np.array([0, 7, 250_000])[:count], np.array([9, 30, 250_003])[:count]
            for g in (c, a, b, a, c):
                got = []
                for mode in (1, 2):
                    params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=2, G=3, R=40, walk_mode=mode)
                    beta, st = pw.pw_query_batch(g.handle, s, t, 0.3, 5, seeds[:count], params)
                    assert np.all(st == 0)
                    got.append(beta)
                np.testing.assert_array_equal(got[0], got[1])


@pytest.mark.parametrize("large,small", [(200_000, 20_001), (500_000, 420_000)])
def test_servers_of_two_graphs(pw, large, small):
    """Two live servers whose kernels are one function with different shared
    memory (25 and 9 KB, 62.5 and 52.5 KB): the first goes on after the second's
    creation, and after the idle time that ends its kernel."""
    import time

    graphs = [cycle_graph(large), cycle_graph(small)]
    params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=2, G=3, R=40)
    with pw.Graph(graphs[0].row_ptr, graphs[0].col_idx) as a, pw.Graph(graphs[1].row_ptr, graphs[1].col_idx) as b:
        servers = []
        try:
            for g in (a, b):
                servers.append(pw.pw_server_create(g.handle, params, 1 << 20))
                for g2, srv in zip((a, b), servers):
                    for i in range(2):
                        ticket = pw.pw_server_submit(srv, i, 1000 + i, 0.3, 9, 5 + i)
                        pw.pw_server_drain(srv, 60000)
                        want = pw.pw_query(g2.handle, i, 1000 + i, 0.3, 9, 5 + i, params)
                        assert pw.pw_server_poll(srv, ticket)[1] == want
                        time.sleep(0.05)
        finally:
            for srv in servers:
                pw.pw_server_destroy(srv)


@pytest.mark.parametrize("graph_fn", [lambda: er_cycle(2000, 12 / 1999, 0), lambda: barabasi_albert(2000, 5, 3)])
def test_series_alone_and_in_a_pass(pw, graph_fn):
    """Ordinary rows of more than 4 entries: a query's bits are the same in passes
    of 4, 8, 16 and 32 columns."""
    host = graph_fn()
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for seed in range(4):
            s, t = uniform_pairs(host.n, 32, 60 + seed)
            for L in (7, 50, 200):
                want = pw.pw_series_batch(g.handle, s, t, L)
                for size in (1, 3, 8, 13):
                    got = np.concatenate([pw.pw_series_batch(g.handle, s[i : i + size], t[i : i + size], L)
                                          for i in range(0, 32, size)])
                    np.testing.assert_array_equal(got, want)


def test_ranked_records_need_not_fit(pw):
    """A graph that fits device memory, but not its ranked form beside it, loads
    and gives the same estimates."""
    import torch

    from pw_inputs import rmat_native

    host = rmat_native(18, 80, (0.57, 0.19, 0.19, 0.05), 6)
    assert 4 * host.nnz + 16 * host.n > 64 << 20 and host.n <= 1 << 21
    s, t = uniform_pairs(host.n, 3, 71)
    seeds = query_seeds(3, 72)

    def estimates(g):
        beta, st = pw.pw_query_batch(g.handle, s, t, 0.3, 21, seeds)
        assert np.all(st == 0)
        return beta

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    for _ in range(2):  # the second load finds the kernels loaded
        before = free()
        with pw.Graph(host.row_ptr, host.col_idx, flags=pw.LOAD_NO_CONNECTIVITY) as g:
            used = before - free()
            want = estimates(g)
    extra = 8 * host.nnz // 3 + 16 * host.n
    fill = torch.empty(free() - (used - extra // 3), dtype=torch.uint8, device="cuda")
    try:
        assert free() < used
        with pw.Graph(host.row_ptr, host.col_idx, flags=pw.LOAD_NO_CONNECTIVITY) as g:
            np.testing.assert_array_equal(estimates(g), want)
    finally:
        del fill
        torch.cuda.empty_cache()


def test_series_replayed_passes(pw, oracle_lib):
    """Groups of several passes on a small graph run as one captured pass that is
    replayed, also for a last pass of fewer queries and for a second group: each
    query's bits are those of a call of its own."""
    from oracle import exact

    host = er_cycle(200, 8 / 199, 0)
    count = 150
    s, t = uniform_pairs(host.n, count, 17)
    t[5] = s[5]
    L = np.tile(np.array([70, 64, 3], np.int32), count // 3)  # replayed (33 and more of each), replayed, not
    L[3:21] = 70
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for _ in range(2):
            got = pw.pw_series_batch(g.handle, s, t, L)
            alone = [pw.pw_series_batch(g.handle, s[i : i + 1], t[i : i + 1], L[i : i + 1])[0] for i in range(count)]
            np.testing.assert_array_equal(got, alone)
        assert got[5] == 0.0
        for length in (64, 70):
            at = np.flatnonzero(L == length)
            assert at.size > 32
            want = exact.series_beta_many(host.row_ptr, host.col_idx, host.n, s[at], t[at], length)
            np.testing.assert_allclose(got[at], want, rtol=1e-9, atol=0)


@pytest.mark.parametrize("n", [8191, 8192, 8193, 16383, 16384, 16385, 135_104, 135_105, 278_528, 278_529])
def test_team_limits(pw, n):
    """Node counts on both sides of the team kernel's limits: builds through pools
    (teams of four below 8,192 nodes, of eight below 16,384, where the pools leave
    shared memory), two tables a block up to 135,104, and a block per probe beyond
    278,528; probes of 3 tiles (teams of four where they fit) and of 10 (eight)."""
    host = cycle_graph(n)
    s, t = np.array([0, 1, n - 1]), np.array([5, n // 2, n - 4])
    seeds = query_seeds(3, n)
    with pw.Graph(host.row_ptr, host.col_idx) as g:
        for R in (96, 300):
            got = []
            for mode in (1, 2):
                params = pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=2, G=11, R=R, walk_mode=mode)
                beta, st = pw.pw_query_batch(g.handle, s, t, 0.3, 9, seeds, params)
                assert np.all(st == 0)
                got.append(beta)
            np.testing.assert_array_equal(got[0], got[1])
