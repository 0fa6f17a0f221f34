"""Performance cases of the library: what a program that uses it has it compute, over the range of sizes that it meets.

Each case loads one synthetic undirected graph (Erdos-Renyi plus ring, preferential attachment, R-MAT, or a 2-D grid
with 5 % of its edges deleted: the families of the tests and the benchmark), keeps its handle (and its server, where
there is one) as a program would, and runs one call with queries that depend on the seed alone: node pairs uniform over
the graph, relative errors in [0.05, 0.2], walk lengths of 8 to 2000 steps.  The handles are used as loaded, with the
library's own choice of kernels (no autotuning, whose timed choice can differ between runs).
"""

import functools
import math
import weakref

import numpy as np
import torch

from paper_2512_05460_gb300 import probewalk as pw

DEV = "cuda"
M32 = 0xFFFFFFFF


def listed():
    return [
        # one interactive query on a small network: launches and latency are all there is
        _case("one_small", "query", "er", 200, 1, 0.2, 0.2, 32),
        # a small batch on the same network (the tiny reference configuration's 64 queries)
        _case("batch_small", "host", "er", 200, 64, 0.2, 0.2, 32),
        # one interactive query on a social-network-like graph
        _case("one_social", "query", "ba", 100_000, 1, 0.1, 0.1, 200),
        # the benchmark's batch on that graph, inputs on the device; a count that is no round number
        _case("batch_social", "device", "ba", 100_000, 75, 0.1, 0.1, 200),
        # a batch of uneven queries on a graph whose records exceed L2 (R-MAT 2^20)
        _case("batch_rmat", "device", "rmat", 1 << 20, 16, 0.05, 0.2, 500),
        # R-MAT beyond the sizes whose probe vector fits on chip: walks that gather from DRAM
        _case("batch_rmat_large", "device", "rmat", 1 << 22, 5, 0.1, 0.2, 1000),
        # a road-network-like graph: local walks, long mixing
        _case("batch_grid", "host", "grid", 2000 * 2000, 24, 0.05, 0.2, 2000),
        # budget adapted to each query's variance, on a graph with an odd node count
        _case("adaptive_social", "host", "ba", 20_001, 33, 0.1, 0.2, 60, "adaptive"),
        # unknown mixing time: the walk length doubles until the estimate stabilises
        _case("stabilized_social", "stabilized", "ba", 100_000, 24, 0.1, 0.1, 256),
        # requests served by continuous batching: a burst through the server
        _case("serve_social", "server", "ba", 20_001, 64, 0.1, 0.2, 100),
        # the deterministic series as a reference for a full group of 32 queries
        _case("series_social", "series", "ba", 100_000, 32, 0.1, 0.1, 200),
        # ... and for a few queries on a grid
        _case("series_grid", "series", "grid", 1000 * 1000, 5, 0.1, 0.1, 301),
    ]


def _case(name, entry, graph, n, count, eps_lo, eps_hi, L, budget="pilot"):
    c = {"entry": entry, "graph": graph, "n": n, "count": count, "eps_lo": eps_lo, "eps_hi": eps_hi, "L": L, "budget": budget}
    return {"name": name, **c} if name else c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choice(["query", "host", "host", "device", "device", "noalloc", "stabilized", "server", "series", "blocks"])
    graph = rng.choice(["er", "ba", "ba", "rmat", "grid"])
    n = {"er": (20, 400), "ba": (1_000, 100_000), "rmat": (1 << 12, 1 << 20), "grid": (30 * 30, 1500 * 1500)}[graph]
    n = _log(rng, *n)
    L = _log(rng, 8, {"er": 100, "ba": 300, "rmat": 500, "grid": 1500}[graph])
    budget = rng.choice(["pilot", "pilot", "pilot", "fixed", "scaled", "adaptive"])
    if entry in ("server", "blocks") and budget == "adaptive":
        budget = "pilot"  # budgets fixed in advance only
    lo, hi = rng.choice([(0.05, 0.2), (0.1, 0.1), (0.2, 0.2), (0.1, 0.2)])
    count = 1 if entry in ("query", "blocks") else _log(rng, 1, 30 if entry == "noalloc" else 70)  # noalloc: 64 MiB of scratch
    c = _case(None, entry, graph, n, count, lo, hi, L, budget)
    if entry == "series":
        c["L"] = min(L, 300)
    most = max(work(x)["flops"] for x in listed() if (x["entry"] == "series") == (entry == "series")) / 2
    while work(c)["flops"] > most and c["count"] > 1:
        c["count"] = max(1, c["count"] // 2)
    return c


# ---- graphs --------------------------------------------------------------------------------------------------------


def _component(n, key):
    """Nodes of the largest connected component of the edges `key` (row * n + col, both directions)."""
    row, col = key // n, key % n
    label = torch.arange(n, device=DEV)
    while True:
        low = label.scatter_reduce(0, row, label[col], "amin")
        low = torch.minimum(low, label.scatter_reduce(0, label[row], low[row], "amin"))
        for _ in range(3):
            low = low[low]
        if torch.equal(low, label):
            break
        label = low
    size = torch.bincount(label, minlength=n)
    return label == size.argmax()


@functools.lru_cache(maxsize=4)
def _csr(graph, n):
    """(row_ptr, col_idx) of the case's graph, on the host."""
    gen = torch.Generator(DEV).manual_seed(1)

    def rand(*shape):
        return torch.rand(*shape, device=DEV, generator=gen, dtype=torch.float64)

    if graph == "er":
        ij = torch.triu_indices(n, n, 1, device=DEV)
        ij = ij[:, rand(ij.shape[1]) < 8 / (n - 1)]
        ring = torch.arange(n, device=DEV)
        u, v = torch.cat([ij[0], ring]), torch.cat([ij[1], (ring + 1) % n])
    elif graph == "ba":  # every new node links to the ends of m=5 places drawn from all earlier edges' ends
        m = 5
        ij = torch.triu_indices(m + 1, m + 1, 1, device=DEV)
        first = ij.shape[1]
        new = torch.arange(m + 1, n, device=DEV).repeat_interleave(m)
        before = first + (new - m - 1) * m
        place = (rand(new.numel()) * 2 * before).long()  # 2e: edge e's source, 2e + 1: its target
        place = torch.cat([2 * torch.arange(first, device=DEV) + 1, place])
        src = torch.cat([ij[0], new])
        while True:  # a target's place leads to the place that target was drawn from
            to = torch.where((place % 2 == 1) & (place // 2 >= first), place[place // 2], place)
            if torch.equal(to, place):
                break
            place = to
        dst = torch.where(place % 2 == 0, src[place // 2], ij[1][(place // 2).clamp(max=first - 1)])
        dst[:first] = ij[1]
        u, v = src, dst
    elif graph == "rmat":
        scale = max(2, (n - 1).bit_length())
        n = 1 << scale
        u = torch.zeros(16 * n, dtype=torch.int64, device=DEV)
        v = torch.zeros_like(u)
        for _ in range(scale):
            r = rand(u.numel())
            u = 2 * u + (r >= 0.76)
            v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    else:
        side = math.isqrt(n)
        n = side * side
        at = torch.arange(n, device=DEV).reshape(side, side)
        u = torch.cat([at[:, :-1].reshape(-1), at[:-1].reshape(-1)])
        v = torch.cat([at[:, 1:].reshape(-1), at[1:].reshape(-1)])
        keep = rand(u.numel()) >= 0.05
        u, v = u[keep], v[keep]
    ok = u != v
    key = torch.unique(torch.cat([u[ok] * n + v[ok], v[ok] * n + u[ok]]))
    if graph in ("rmat", "grid"):
        keep = _component(n, key)
        new_id = torch.cumsum(keep, 0) - 1
        row, col = key // n, key % n
        inside = keep[row]
        n = int(keep.sum())
        row, col = new_id[row[inside]], new_id[col[inside]]
    else:
        row, col = key // n, key % n
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    out = row_ptr.cpu().numpy(), col.to(torch.int32).cpu().numpy()
    del u, v, key, row, col
    torch.cuda.empty_cache()
    return out


class _Server:
    """A server on a loaded graph, stopped with its last user."""

    def __init__(self, graph, params):
        self.graph = graph
        self.handle = pw.pw_server_create(graph.handle, params, 1 << 28)

    def __del__(self):
        pw.pw_server_destroy(self.handle)


# Handles are kept while a state that uses them lives, as a program keeps its loaded graph between calls.
_graphs = weakref.WeakValueDictionary()
_servers = weakref.WeakValueDictionary()


def _graph(case):
    key = case["graph"], case["n"]
    g = _graphs.get(key)
    if g is None:
        # the generators return connected graphs, so the program skips the O(n + m) check
        g = _graphs[key] = pw.Graph(*_csr(*key), flags=pw.LOAD_NO_CONNECTIVITY)
    return g


# ---- calls ---------------------------------------------------------------------------------------------------------


def _params(case):
    if case["budget"] == "fixed":
        return pw.make_params(budget_mode=pw.PW_BUDGET_FIXED, B=3, G=9, R=200)
    if case["budget"] == "scaled":
        return pw.make_params(budget_mode=pw.PW_BUDGET_SCALED, c_B=1e-3, c_R=1e-4, R_max=500, delta=0.05)
    return pw.make_params(budget_mode=pw.PW_BUDGET_ADAPTIVE if case["budget"] == "adaptive" else pw.PW_BUDGET_PILOT)


def _queries(case, seed, n):
    rng = np.random.default_rng(seed)
    s = rng.integers(0, n, case["count"], dtype=np.int64)
    t = rng.integers(0, n - 1, case["count"], dtype=np.int64)
    t += t >= s
    eps = rng.uniform(case["eps_lo"], case["eps_hi"], case["count"])
    L = np.full(case["count"], case["L"], np.int32)
    seeds = rng.integers(0, 2**63 - 1, case["count"], dtype=np.int64).astype(np.uint64)
    return s, t, eps, L, seeds


def prepare(case, seed):
    g = _graph(case)
    q = _queries(case, seed, g.n)
    state = {"case": case, "graph": g, "q": q, "params": _params(case)}
    if case["entry"] in ("device", "noalloc"):
        state["dev"] = [torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a).to(DEV) for a in q]
        state["beta"] = torch.zeros(case["count"], dtype=torch.float64, device=DEV)
        state["status"] = torch.zeros(case["count"], dtype=torch.int32, device=DEV)
    if case["entry"] == "server":
        key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
        srv = _servers.get(key)
        if srv is None:
            srv = _servers[key] = _Server(g, state["params"])
        state["server"] = srv
    return state


def run(state):
    case, g, params = state["case"], state["graph"].handle, state["params"]
    s, t, eps, L, seeds = state["q"]
    entry = case["entry"]
    if entry == "query":
        return pw.pw_query(g, int(s[0]), int(t[0]), float(eps[0]), int(L[0]), int(seeds[0]), params)
    if entry == "blocks":  # the second half of a query's blocks, as one of two ranks runs it
        lo, hi = _block_range(case)
        return pw.pw_query_blocks(g, int(s[0]), int(t[0]), float(eps[0]), int(L[0]), lo, hi, int(seeds[0]), params)
    if entry in ("device", "noalloc"):
        call = pw.pw_query_batch_device if entry == "device" else pw.pw_query_batch_noalloc
        call(g, case["count"], *state["dev"], state["beta"], state["status"], params)
        return state["beta"], state["status"]
    if entry == "stabilized":
        return pw.pw_query_stabilized(g, s, t, eps, max(2, case["L"]), seeds, params)
    if entry == "series":
        return pw.pw_series_batch(g, s, t, L)
    if entry == "server":
        srv = state["server"].handle
        for i in range(case["count"]):
            pw.pw_server_submit(srv, int(s[i]), int(t[i]), float(eps[i]), int(L[i]), int(seeds[i]))
        pw.pw_server_drain(srv)
        tickets, beta, status, _ = pw.pw_server_collect(srv, case["count"])
        order = np.argsort(tickets)
        return beta[order], status[order]
    return pw.pw_query_batch(g, s, t, eps, L, seeds, params)


# ---- work ----------------------------------------------------------------------------------------------------------


def _blocks(case):
    return {"fixed": 9, "scaled": 24}.get(case["budget"], 37)  # G


def _block_range(case):
    return _blocks(case) // 2, _blocks(case)


def work(case):
    """Bytes: the CSR arrays and the queries read once, the results written once.  Operations: per node visited, a
    quarter of a Philox block (10 rounds of two multiplications and four exclusive-ors), the neighbour's index and one
    addition; per series step, an addition per entry and query, one multiplication and one addition per node and query.
    The replicas of a pilot budget follow the data: typical ones of the family stand for them."""
    n, count, L = case["n"], case["count"], case["L"]
    entries = {"er": 10, "ba": 10, "rmat": 29, "grid": 3.8}[case["graph"]] * n
    bytes_ = 8 * (n + 1) + 4 * entries + 48 * count
    if case["entry"] == "series":
        return {"bytes": float(bytes_), "flops": float(count * (L + 1) * (entries + 2 * n))}
    lo, hi = case["eps_lo"], case["eps_hi"]
    probes = 37 * 0.5 / (lo * hi)  # the mean of 1 / eps^2 over [lo, hi]
    replicas = {"er": 200, "ba": 800, "rmat": 900, "grid": 50}[case["graph"]]
    if case["budget"] == "fixed":
        probes, replicas = 27, 200
    if case["budget"] == "scaled":
        probes, replicas = 24 * 1e-3 * 448 / (lo * hi), 500
    if case["entry"] == "blocks":
        probes /= 2
    if case["entry"] == "stabilized":
        L = min(L, 16)  # most queries stop by then
    return {"bytes": float(bytes_), "flops": float(count * probes * replicas * 2 * (L + 1) * 17)}


# ---- the same estimator in 64 bits, in plain torch -----------------------------------------------------------------


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & M32, seed >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # the low 64 bits, as int64
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _probes(n, seed, k, tag):
    """z of every node for the probes k: [len(k), n] in {-1, 0, 1}."""
    k = k[:, None]
    zero = torch.zeros_like(k)
    a0, a1, b0, b1 = _philox(k, zero, zero, zero + tag, seed)

    def mod(lo, hi, p):  # (lo + 2^32 hi) mod p
        return ((hi % p) * ((1 << 32) % p) + lo % p) % p

    p = (1 << 31) - 1
    a, b = 1 + mod(a0, a1, p - 1), mod(b0, b1, p)
    keys = [w for j in range(3) for w in _philox(k, zero + 1, zero + j, zero + tag, seed)]
    coin = _philox(k, zero + 2, zero, zero + tag, seed)[0]
    r = zero + 1 if n & 1 else 2 * (coin & 1)
    bits = max(2, (n - 1).bit_length())
    bits = 4 if bits == 3 else bits
    hi, lo = (bits + 1) // 2, bits // 2

    def permute(x):
        left, right = x >> lo, x & ((1 << lo) - 1)
        for i in range(12 if bits <= 4 else 8):
            y = ((right ^ keys[i]) * 0x9E3779B1) & M32
            y = ((y ^ (y >> 16)) * 0x85EBCA6B) & M32
            left, right = right, left ^ (y >> (32 - (lo if i & 1 else hi)))
        return (left << lo) | right

    dom = permute(torch.arange(1 << bits, device=DEV)[None, :].expand(k.shape[0], -1))
    pi = dom[:, :n]
    while bool((pi >= n).any()):
        pi = torch.where(pi >= n, dom.gather(1, pi), pi)
    sign = 1 - 2 * ((((a * (pi >> 1) + b) % p) + pi) & 1)
    return torch.where(pi >= n - r, 0, sign)


def _sums(g, s, t, L, seed, R, ks, walk_tag, probe_tag):
    """(S1, S2) of the probes ks in 64 bits."""
    row_ptr, col, n = g
    deg = row_ptr[1:] - row_ptr[:-1]
    inv = 1.0 / deg.double()
    S1, S2 = [], []
    per = max(1, min(8_000_000 // (2 * R), 100_000_000 // n))
    for at in range(0, ks.numel(), per):
        k = ks[at : at + per]
        z = _probes(n, seed, k, probe_tag).to(torch.int8)
        which = torch.arange(k.numel(), device=DEV).repeat_interleave(R)[None, :]
        pair = (k[:, None] * R + torch.arange(R, device=DEV)[None, :]).reshape(-1)
        walk = torch.stack([2 * pair, 2 * pair + 1])
        v = torch.tensor([[s], [t]], device=DEV).expand_as(walk)
        total = z[which, v].double() * inv[v]
        zero = torch.zeros_like(walk)
        for i in range(1, L + 1):
            if i == 1 or i % 4 == 0:
                words = _philox(walk & M32, walk >> 32, zero + i // 4, zero + walk_tag, seed)
            v = col[row_ptr[v] + ((words[i % 4] * deg[v]) >> 32)]
            total += z[which, v].double() * inv[v]
        U = (total[0] - total[1]).reshape(-1, R)
        S1.append(U.sum(1))
        S2.append((U * U).sum(1))
    return torch.cat(S1), torch.cat(S2)


class _TooLong(Exception):
    pass


def _ceil(x):
    return int(math.ceil(x * (1 - 1e-12)))


def _estimate(g, case, s, t, eps, L, seed, left):
    """Algorithm 1 for one query: the G block means and their median.  `left`: node visits still affordable."""
    row_ptr, _, n = g
    ds, dt = (int(row_ptr[v + 1] - row_ptr[v]) for v in (s, t))
    inv = 1 / ds + 1 / dt
    theta0 = (1 - eps / 2) * inv * inv / 8
    G, kind, B_max = _blocks(case), case["budget"], 0
    if kind == "fixed":
        B, R = 3, 200
    elif kind == "scaled":
        d_min = int((row_ptr[1:] - row_ptr[:-1]).min())
        B = max(1, _ceil(1e-3 * 448 / eps**2))
        R = min(500, max(2, _ceil(1e-4 * (128 * (L + 1) ** 2 / (d_min**2 * (1 - eps / 2) * inv * inv)))))
    else:
        B = max(1, _ceil(0.5 / eps**2))
        S1, S2 = _sums(g, s, t, L, seed, 32, torch.arange(64, device=DEV), 2, 4)
        sigma2 = float(((S2 - S1 * S1 / 32) / 31).mean())
        theta = max(float(((S1 * S1 - S2) / (32 * 31)).mean()), theta0)
        R = min(4096, 32 * math.ceil(max(2, _ceil(4 * sigma2 / theta)) / 32))
        if kind == "adaptive":
            B_max, B = 2 * B, (B + 3) // 4

    def q_values(lo, hi):
        left[0] -= (hi - lo) * (2 * R * (L + 1) + n)
        if left[0] < 0:
            raise _TooLong
        S1, S2 = _sums(g, s, t, L, seed, R, torch.arange(lo, hi, device=DEV), 1, 3)
        return (S1 * S1 - S2) / (R * (R - 1.0))

    if case["entry"] == "blocks":
        lo, hi = _block_range(case)
        return q_values(lo * B, hi * B).reshape(-1, B).mean(1), None
    Q = q_values(0, G * B)
    if B_max:
        theta = max(float(Q.mean()), theta0)
        want = _ceil(math.pi / 2 * 9 * float(Q.var()) / theta**2 / (G * eps * eps))
        more = min(max(want, B), B_max)
        if more > B:
            Q, B = torch.cat([Q, q_values(G * B, G * more)]), more
    return None, float(Q.reshape(G, B).mean(1).quantile(0.5))


def _level_seed(seed, L):
    w = _philox(*(torch.tensor(x) for x in (L, 0, 0, 0x57AB)), seed)
    return int(w[0]) | (int(w[1]) << 32)


def _series(g, s, t, L):
    row_ptr, col, n = g
    deg = (row_ptr[1:] - row_ptr[:-1]).double()
    A = torch.sparse_csr_tensor(row_ptr, col, torch.ones(col.numel(), dtype=torch.float64, device=DEV), (n, n))
    cols = torch.arange(s.size, device=DEV)
    x = torch.zeros(n, s.size, dtype=torch.float64, device=DEV)
    s, t = (torch.from_numpy(v).to(DEV) for v in (s, t))
    x[s, cols] = 1 / deg[s]
    x[t, cols] = -1 / deg[t]
    h = x.clone()
    for _ in range(L):
        x = (A @ x) / deg[:, None]
        h += x
    return ((h * h).sum(0) - h.sum(0) ** 2 / n).cpu().numpy()


def exact(case, seed):
    """What run() returns, with every sum and quotient in 64 bits; None where that takes too long."""
    if case["entry"] != "series" and work(case)["flops"] / 17 > 1e10:
        return None
    row_ptr, col = (torch.from_numpy(a).to(DEV) for a in _csr(case["graph"], case["n"]))
    n = row_ptr.numel() - 1
    g = row_ptr, col.long(), n
    s, t, eps, L, seeds = _queries(case, seed, n)
    if case["entry"] == "series":
        return _series(g, s, t, case["L"])
    left = [6e9]
    beta, stop = np.zeros(s.size), np.zeros(s.size, np.int32)
    try:
        for i in range(s.size):
            q = int(s[i]), int(t[i]), float(eps[i])
            if case["entry"] == "stabilized":
                level, last, most = 1, None, max(2, case["L"])
                while True:
                    beta[i] = _estimate(g, case, *q, level, _level_seed(int(seeds[i]), level), left)[1]
                    stop[i] = level
                    if level >= most or (last is not None and abs(beta[i] - last) <= q[2] / 2 * abs(beta[i])):
                        break
                    level, last = min(2 * level, most), beta[i]
                continue
            means, beta[i] = _estimate(g, case, *q, case["L"], int(seeds[i]), left)
            if means is not None:
                return means.cpu().numpy()
    except _TooLong:
        return None
    if case["entry"] == "query":
        return float(beta[0])
    if case["entry"] == "stabilized":
        return beta, None, None
    return beta, None
