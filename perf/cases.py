"""Workloads that a user of this library runs, through its public entry points.

``listed()`` names the standing cases, ``draw(rng)`` gives others of the same
ranges, ``prepare`` makes what a program has in hand before the call (inputs
on the GPU, or resident graphs), ``run`` is one pass, ``work`` the bytes that
a pass cannot do without, and ``exact`` the values of a pass by plain torch in
64 bits (every triangle or clique enumerated).

Graphs are erased Chung-Lu power-law graphs with heavy-tailed weights, the
recipe of the benchmark and the tests, drawn on the device from the seed.
"""
import math

import numpy as np
import torch

import paper_1910_00692_gb300 as wt

DEV = "cuda"


# ---------------------------------------------------------------------------
# The cases.
# ---------------------------------------------------------------------------
def listed():
    return [
        # One small graph in host arrays, built, asked once and dropped: the
        # smallest request, where launches and latency count.
        {"name": "build_tiny_host", "kind": "build", "n": 2000, "m": 20000, "gamma": 2.1, "dmax": 200.0,
         "weights": "counts", "where": "host", "ps": "1", "k": 100},
        # Real-valued weights (similarities) on a graph of a million edges,
        # neither size a round number.
        {"name": "build_real_1m", "kind": "build", "n": 50021, "m": 1000003, "gamma": 2.1, "dmax": 11181.0,
         "weights": "real", "where": "device", "ps": "2", "k": 1000},
        # The 2e7-edge configuration: build from device arrays, then a query.
        {"name": "build_20m", "kind": "build", "n": 1000000, "m": 20000000, "gamma": 2.1, "dmax": 50000.0,
         "weights": "zipf", "where": "device", "ps": "1", "k": 1000},
        # The billion-edge configuration, the library's headline.
        {"name": "build_1b", "kind": "build", "n": 50000000, "m": 1000000000, "gamma": 2.0, "dmax": 50000.0,
         "weights": "zipf", "where": "device", "ps": "1", "k": 1000},
        # The four exact means on the resident 2e7-edge graph, device results.
        {"name": "query_20m", "kind": "query", "n": 1000000, "m": 20000000, "gamma": 2.1, "dmax": 50000.0,
         "weights": "zipf", "ps": "-inf,1,2,inf", "k": 1000},
        # A serving-pool graph (2e8 edges): the minimum, which prunes least,
        # and the arithmetic mean.
        {"name": "query_200m", "kind": "query", "n": 10000000, "m": 200000000, "gamma": 2.1, "dmax": 50000.0,
         "weights": "zipf", "ps": "-inf,1", "k": 1000},
        # Harmonic and geometric means and p = 3 (fp64 and product keys).
        {"name": "query_means_5m", "kind": "query", "n": 250000, "m": 5000000, "gamma": 2.1, "dmax": 25000.0,
         "weights": "zipf", "ps": "-1,0,3", "k": 500},
        # Weighted edge sampling with many draws.
        {"name": "sample_edges_20m", "kind": "edges", "n": 1000000, "m": 20000000, "gamma": 2.1, "dmax": 50000.0,
         "weights": "zipf", "ps": "1", "k": 1000, "draws": 1000000},
        # Weighted wedge sampling.
        {"name": "sample_wedges_2m", "kind": "wedges", "n": 100000, "m": 2000000, "gamma": 2.1, "dmax": 15811.0,
         "weights": "zipf", "ps": "1", "k": 1000, "draws": 1000000},
        # Top 5-cliques of a small dense graph by edge sampling.
        {"name": "cliques5_979", "kind": "cliques", "n": 979, "m": 29000, "gamma": 2.1, "dmax": 489.5,
         "weights": "events", "ps": "1", "k": 1000, "q": 5, "draws": 10000},
        # One batched call over 1,024 resident graphs of uneven sizes.
        {"name": "batch_1024", "kind": "batch", "count": 1024, "n_hi": 20000},
        # A burst of mixed requests to the server over a pool of three graphs.
        {"name": "serve_burst_512", "kind": "serve", "requests": 512, "m": 20000000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "query", "query", "edges", "wedges", "cliques", "batch", "serve"])
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 16, 1500), "n_hi": _log(rng, 1000, 20000)}
    if kind == "serve":
        return {"kind": kind, "requests": _log(rng, 8, 512), "m": _log(rng, 200000, 20000000)}
    if kind == "cliques":
        n, q = rng.randint(200, 979), rng.choice([4, 5])
        return {"kind": kind, "n": n, "m": int(n * rng.uniform(8, 30 if n > 500 else 16)), "gamma": 2.1,
                "dmax": n / 2.0, "weights": "events", "ps": rng.choice(["1", "2"]), "k": _log(rng, 10, 1000), "q": q,
                "draws": rng.choice([_log(rng, 300, 30000), -1])}
    hi = {"build": 400000000, "query": 200000000, "edges": 40000000, "wedges": 10000000}[kind]
    m = _log(rng, 5000, hi) | rng.randint(0, 1)
    n = max(200, int(m / rng.uniform(8, 30)))
    c = {"kind": kind, "n": n, "m": m, "gamma": rng.choice([2.0, 2.1, 2.2]),
         "dmax": float(min(n - 1, int(50000 * math.sqrt(m / 2e7)), 50000)),
         "weights": rng.choice(["zipf", "zipf", "counts"]), "k": _log(rng, 10, 5000)}
    if kind == "build":
        c["where"] = rng.choice(["host", "device", "device"]) if m < 3000000 else "device"
        c["weights"] = rng.choice(["zipf", "zipf", "counts", "real"])
        c["ps"] = rng.choice(["-inf", "1", "2", "inf"])
    elif kind == "query":
        c["ps"] = rng.choice(["-inf,1", "1,2", "2,inf", "inf,1", "-inf,1,2,inf"]) if m > 5000000 else \
            rng.choice(["-1,0", "0,1,2", "-inf,3", "1,2", "-inf,1,2,inf", "-2,0.5"])
    else:
        c["ps"] = rng.choice(["0", "1", "2"]) if kind == "edges" else rng.choice(["1", "1", "2"])
        c["draws"] = _log(rng, 1000, 2000000)
        if kind == "wedges":
            c.update(weights="counts", n=n & ~1, k=c["k"] & ~1, draws=c["draws"] & ~1)
    return c


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _offsets(ns, ms, a, dmax):
    """i0 of each graph's degree profile dmax (1 + x / i0)^-a on [0, n), whose
    integral is 2 m (bisection; dmax is reached at x = 0)."""
    lo, hi = np.full(ns.shape, 1e-9), np.full(ns.shape, 1e12)
    for _ in range(120):
        mid = np.sqrt(lo * hi)
        if abs(a - 1) < 1e-9:
            total = dmax * mid * np.log1p(ns / mid)
        else:
            total = dmax * mid / (1 - a) * np.expm1((1 - a) * np.log1p(ns / mid))
        low = total < 2.0 * ms
        lo, hi = np.where(low, mid, lo), np.where(low, hi, mid)
    return hi


def _pairs(ns, ms, gamma, dmax, gen):
    """Endpoints of simple Chung-Lu graphs, graph after graph: exactly ms[g]
    distinct pairs of graph g, in the order drawn, either endpoint first."""
    ns, ms = np.asarray(ns, np.int64), np.asarray(ms, np.int64)
    a = 1.0 / (gamma - 1.0)
    i0 = _offsets(ns.astype(float), ms.astype(float), a, np.asarray(dmax, float))
    bits = int(int(ns.max()) ** 2 - 1).bit_length()
    factor = 1.15
    while True:
        counts = (ms * factor).astype(np.int64) + 64
        u = torch.empty(int(counts.sum()), dtype=torch.int32, device=DEV)
        v = torch.empty_like(u)
        single = len(ns) == 1
        cnt = torch.as_tensor(counts, device=DEV)
        gid = None if single else torch.repeat_interleave(torch.arange(len(ns), device=DEV), cnt)
        par = torch.as_tensor(np.stack([i0, ns.astype(float)]), device=DEV)
        for at in range(0, u.numel(), 1 << 27):
            end = min(u.numel(), at + (1 << 27))
            off, nn = (float(i0[0]), float(ns[0])) if single else (par[0][gid[at:end]], par[1][gid[at:end]])
            for out in (u, v):
                x = torch.rand(end - at, dtype=torch.float64, device=DEV, generator=gen)
                span = math.log1p(nn / off) if single else torch.log1p(nn / off)
                if abs(a - 1) < 1e-9:
                    x = off * torch.expm1(x * span)
                else:
                    top = math.expm1((1 - a) * span) if single else torch.expm1((1 - a) * span)
                    x = off * torch.expm1(torch.log1p(x * top) / (1 - a))
                x = x.floor_().clamp_(min=0)
                out[at:end] = (x.clamp_(max=nn - 1) if single else torch.minimum(x, nn - 1)).to(torch.int32)
                del x
        keys = torch.minimum(u, v).to(torch.int64)
        nn = int(ns[0]) if single else par[1][gid].to(torch.int64)
        keys.mul_(nn).add_(torch.maximum(u, v))
        if not single:
            keys.add_(gid << bits)
        keys, at = torch.sort(keys, stable=True)
        first = torch.ones(keys.numel(), dtype=torch.bool, device=DEV)
        first[1:] = keys[1:] != keys[:-1]
        del keys
        keep = torch.empty_like(first)
        keep[at] = first
        del at, first
        keep &= u != v
        if single:
            got = int(keep.sum())
            if got >= int(ms[0]):
                return u[keep][: int(ms[0])].clone(), v[keep][: int(ms[0])].clone()
        else:
            gk = gid[keep]
            have = torch.bincount(gk, minlength=len(ns))
            want = torch.as_tensor(ms, device=DEV)
            if bool((have >= want).all()):
                start = torch.cumsum(have, 0) - have
                inside = torch.arange(gk.numel(), device=DEV) - start[gk] < want[gk]
                return u[keep][inside], v[keep][inside]
        factor *= 1.5


def _zipf(m, s, cap, gen):
    cdf = torch.cumsum(torch.arange(1, cap + 1, dtype=torch.float64, device=DEV) ** -s, 0)
    cdf /= cdf[-1].clone()
    out = torch.empty(m, dtype=torch.int32, device=DEV)
    for at in range(0, m, 1 << 27):
        end = min(m, at + (1 << 27))
        x = torch.rand(end - at, dtype=torch.float64, device=DEV, generator=gen)
        out[at:end] = torch.searchsorted(cdf, x, right=True, out_int32=True).add_(1).clamp_(max=cap)
    return out


def _weights(m, kind, gen):
    if kind == "zipf":
        return _zipf(m, 2.0, 1000000, gen)
    if kind == "events":
        return _zipf(m, 1.7, 50000, gen)
    if kind == "counts":  # 1 + geometric(0.3), one in a hundred heavy-tailed
        x = torch.rand(m, dtype=torch.float64, device=DEV, generator=gen)
        w = (torch.log1p(-x) / math.log(0.7)).floor_().to(torch.int32) + 1
        heavy = torch.rand(m, device=DEV, generator=gen) < 0.01
        return torch.where(heavy, _zipf(m, 1.5, 10000, gen), w)
    x = torch.randn(m, dtype=torch.float64, device=DEV, generator=gen)  # log-normal similarities
    return torch.exp(x).clamp_(min=1e-6, max=1e6).to(torch.float32)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 101)
    return g


def _edges(case, seed):
    gen = _gen(seed)
    u, v = _pairs([case["n"]], [case["m"]], case["gamma"], [case["dmax"]], gen)
    w = _weights(case["m"], case["weights"], gen)
    if case["m"] > 100000000:
        torch.cuda.empty_cache()  # the draw's temporaries
    return u, v, w


def _batch_edges(case, seed):
    """Sizes and queries of a batch, and its graphs' edges in one array each."""
    c = case["count"]
    rng = np.random.default_rng([c, case["n_hi"]])
    ns = np.exp(rng.uniform(math.log(100), math.log(case["n_hi"]), c)).astype(np.int64)
    ms = np.minimum(10 * ns, ns * (ns - 1) // 2)
    ks = rng.integers(10, 1001, c).astype(np.int32)
    ps = np.array([-math.inf, 1.0, 2.0, math.inf])[rng.integers(0, 4, c)]
    gen = _gen(seed)
    u, v = _pairs(ns, ms, 2.2, np.minimum(ns - 1, np.sqrt(2.0 * ms)), gen)
    w = _weights(int(ms.sum()), "zipf", gen)
    return ns, ms, ps, ks, u, v, w


def _pool(case):
    """The server's graphs (a tenth and a quarter of the largest) and requests."""
    m = case["m"]
    graphs = [dict(n=x // 20, m=x, gamma=2.1, dmax=float(min(x // 20 - 1, int(50000 * math.sqrt(x / 2e7)))),
                   weights="zipf") for x in (m, m // 4, m // 10)]
    r = case["requests"]
    rng = np.random.default_rng([r, m])
    gs = rng.integers(0, 3, r)
    ps = np.array([-math.inf, 1.0, 2.0, math.inf])[rng.integers(0, 4, r)]
    ks = rng.integers(10, 1001, r)
    return graphs, [(int(a), float(b), int(c)) for a, b, c in zip(gs, ps, ks)]


def _ps(case):
    return [float(p) for p in case["ps"].split(",")]


def _outs(case):
    k = case["k"]
    return [(p, torch.full((k, 3), -1, dtype=torch.int32, device=DEV), torch.zeros(k, dtype=torch.float64, device=DEV),
             torch.zeros(1, dtype=torch.int32, device=DEV)) for p in _ps(case)]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": int(seed)}
    if kind == "batch":
        ns, ms, ps, ks, u, v, w = _batch_edges(case, seed)
        at = np.concatenate([[0], np.cumsum(ms)])
        s["graphs"] = [wt.build_csr(int(ns[g]), *(x[at[g]:at[g + 1]] for x in (u, v, w))) for g in range(len(ns))]
        s["ps"], s["ks"] = ps, ks
    elif kind == "serve":
        graphs, s["requests"] = _pool(case)
        s["graphs"] = [wt.build_csr(g["n"], *_edges(g, seed * 3 + i)) for i, g in enumerate(graphs)]
        s["server"] = wt.Server(120 << 30, 256)
        for g in s["graphs"]:
            s["server"].add_graph(g)
    else:
        u, v, w = _edges(case, seed)
        if kind == "build":
            s["uvw"] = tuple(x.cpu().numpy() for x in (u, v, w)) if case["where"] == "host" else (u, v, w)
        else:
            s["graph"] = wt.build_csr(case["n"], u, v, w)
        s["outs"] = _outs(case)
    return s


# ---------------------------------------------------------------------------
# One pass.
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "build":
        g = wt.build_csr(case["n"], *s["uvw"])
        if case["where"] == "host":
            out = [_kept([case["k"]], [wt.topk(g, p, case["k"])]) for p in _ps(case)]
        else:
            for p, t, w, c in s["outs"]:
                wt.topk_device(g, p, case["k"], t, w, c)
            out = [(t, w, c) for _, t, w, c in s["outs"]]
        g.free()
        return out
    if kind == "query":
        for p, t, w, c in s["outs"]:
            wt.topk_device(s["graph"], p, case["k"], t, w, c)
        return [(t, w, c) for _, t, w, c in s["outs"]]
    if kind == "edges":
        return _kept([case["k"]], [wt.sample_topk(s["graph"], _ps(case)[0], case["k"], case["draws"], s["seed"])])
    if kind == "wedges":
        return _kept([case["k"]], [wt.wedge_topk(s["graph"], _ps(case)[0], case["k"], case["draws"], s["seed"])])
    if kind == "cliques":
        ids, w, keys = wt.sample_cliques(s["graph"], case["q"], _ps(case)[0], case["k"], case["draws"], s["seed"])
        out = np.zeros(case["k"], np.int64)
        out[:len(w)] = keys.view(np.int64)
        return *_kept([case["k"]], [(ids, w)]), out
    if kind == "batch":
        return _kept(s["ks"], wt.topk_batch(s["graphs"], s["ps"], s["ks"]))
    server = s["server"]
    tickets = [server.submit(g, p, k) for g, p, k in s["requests"]]
    got = []
    for t, (_, _, k) in zip(tickets, s["requests"]):
        r = server.poll(t, k)
        while r is None:
            r = server.poll(t, k)
        got.append(r[:2])
    return _kept([k for _, _, k in s["requests"]], got)


def _kept(ks, results):
    """The results of queries for ks[i] each, one after another in the
    program's own arrays: ids (-1 past the last), weights (0), and counts."""
    at = np.concatenate([[0], np.cumsum(ks)])
    ids = np.full((int(at[-1]), results[0][0].shape[1]), -1, np.int32)
    weights = np.zeros(int(at[-1]))
    for a, (t, w) in zip(at, results):
        ids[a:a + len(w)], weights[a:a + len(w)] = t, w
    return ids, weights, np.array([len(w) for _, w in results])


def _padded(ks, values):
    """_kept's layout of the values alone."""
    return None, _kept(ks, [(np.full((x.numel(), 3), -1, np.int32), x.cpu().numpy()) for x in values])[1], None


def work(case):
    """Build: the edge list read, the resident graph (48 bytes an edge, 16 a
    vertex) written.  Queries: the three edges (two ids and a weight each) of
    every triangle returned, and the results.  Sampling adds one edge a draw."""
    kind = case["kind"]
    if kind == "batch":
        return {"bytes": case["count"] * 505 * 56, "flops": 0}
    if kind == "serve":
        return {"bytes": case["requests"] * 505 * 56, "flops": 0}
    out = len(_ps(case)) * case["k"] * 56
    if kind == "build":
        return {"bytes": 60 * case["m"] + 16 * case["n"] + out, "flops": 0}
    if kind == "cliques":
        edges = case["m"] if case["draws"] < 0 else min(case["m"], case["draws"])
        return {"bytes": 12 * edges + case["k"] * (4 * case["q"] + 16), "flops": 0}
    if kind in ("edges", "wedges"):
        out += 12 * case["draws"]
    return {"bytes": out, "flops": 0}


# ---------------------------------------------------------------------------
# The values of a pass by enumeration (float64 torch, none of the library).
# ---------------------------------------------------------------------------
def _mean(ws, p):
    x = torch.stack([w.double() for w in ws])
    if p == math.inf:
        return x.amax(0)
    if p == -math.inf:
        return x.amin(0)
    if p == 0:
        return torch.exp(torch.log(x).mean(0))
    top = x.amax(0) if p > 0 else x.amin(0)
    return top * ((x / top) ** p).mean(0) ** (1.0 / p)


def _top_values(n, u, v, w, ps, k, drawn=None):
    """The k largest p-means over the triangles (those with a drawn edge, if
    given), descending, for every p of ps: all wedges at each vertex of lower
    (degree, id) rank, closed by a search in the sorted edges."""
    u, v = u.long(), v.long()
    deg = torch.bincount(torch.cat([u, v]), minlength=n)
    rank = torch.empty(n, dtype=torch.int64, device=DEV)
    rank[torch.sort(deg, stable=True).indices] = torch.arange(n, device=DEV)
    ru, rv = rank[u], rank[v]
    key, at = torch.sort(torch.minimum(ru, rv) * n + torch.maximum(ru, rv))
    w = w[at]
    drawn = None if drawn is None else drawn[at]
    src, dst = key // n, key % n
    ends = torch.searchsorted(src, src, right=True)
    place = torch.arange(key.numel(), device=DEV)
    number = ends - place - 1  # wedges whose lower edge this is
    upto = torch.cumsum(number, 0)
    best = [torch.empty(0, dtype=torch.float64, device=DEV) for _ in ps]
    total, lo, step = int(upto[-1]), 0, 1 << 25
    while lo < total:
        hi = min(total, lo + step)
        x = torch.arange(lo, hi, device=DEV)
        e1 = torch.searchsorted(upto, x, right=True)
        e2 = e1 + 1 + x - (upto[e1] - number[e1])
        want = dst[e1] * n + dst[e2]
        e3 = torch.searchsorted(key, want).clamp_(max=key.numel() - 1)
        ok = key[e3] == want
        if drawn is not None:
            ok &= drawn[e1] | drawn[e2] | drawn[e3]
        ws = [w[e[ok]] for e in (e1, e2, e3)]
        for i, p in enumerate(ps):
            vals = torch.cat([best[i], _mean(ws, p)])
            best[i] = torch.topk(vals, min(k, vals.numel())).values
        lo = hi
    return best


def _drawn_edges(w, p, draws, seed):
    """Which edges weighted sampling draws: word 0 of Philox4x64-10 (counter
    = the draw's index, key = the seed), scaled to the total mass, looked up
    in the cumulative masses of the edges by falling weight (ties by index)."""
    w = w.cpu().numpy().astype(np.uint64)
    order = np.argsort(-w.astype(np.int64), kind="stable")
    cum = np.cumsum(w[order] ** np.uint64(int(p)))
    z = cum[-1]
    gen = np.random.Philox(key=np.array([seed, 0], np.uint64), counter=np.array([2 ** 64 - 1] * 4, np.uint64))
    x = gen.random_raw(4 * draws)[::4]
    low, half = np.uint64(0xFFFFFFFF), np.uint64(32)
    xl, xh, zl, zh = x & low, x >> half, z & low, z >> half
    mid = xh * zl + (xl * zl >> half)
    mid2 = xl * zh + (mid & low)
    t = xh * zh + (mid >> half) + (mid2 >> half)
    marks = np.zeros(w.size, bool)
    marks[order[np.searchsorted(cum, t, side="right")]] = True
    return torch.from_numpy(marks).to(DEV)


def _clique_values(n, u, v, w, q, p, k, drawn):
    adj = torch.zeros((n, n), dtype=torch.bool, device=DEV)
    wt2 = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    mark = torch.zeros((n, n), dtype=torch.bool, device=DEV)
    a, b = torch.minimum(u, v).long(), torch.maximum(u, v).long()
    adj[a, b], wt2[a, b], mark[a, b] = True, w.double(), drawn
    got = adj.nonzero()
    for _ in range(q - 2):
        parts = []
        for c in torch.split(got, max(1, (1 << 29) // n)):
            common = adj[c[:, 0]]
            for j in range(1, c.shape[1]):
                common &= adj[c[:, j]]
            x = common.nonzero()
            parts.append(torch.cat([c[x[:, 0]], x[:, 1:]], 1))
        got = torch.cat(parts)
    pairs = [(i, j) for i in range(q) for j in range(i + 1, q)]
    any_ = torch.stack([mark[got[:, i], got[:, j]] for i, j in pairs]).any(0)
    got = got[any_]
    vals = _mean([wt2[got[:, i], got[:, j]] for i, j in pairs], p)
    return torch.topk(vals, min(k, vals.numel())).values


def exact(case, seed):
    kind = case["kind"]
    if kind == "wedges" or (kind not in ("batch", "serve") and case["m"] > 25000000):
        return None  # three exact mixture draws a sample; too many wedges to list
    if kind == "batch":
        ns, ms, ps, ks, u, v, w = _batch_edges(case, seed)
        at = np.concatenate([[0], np.cumsum(ms)])
        vals = [_top_values(int(ns[g]), *(x[at[g]:at[g + 1]] for x in (u, v, w)), [ps[g]], int(ks[g]))[0]
                for g in range(len(ns))]
        return _padded(ks, vals)
    if kind == "serve":
        graphs, requests = _pool(case)
        ps = [-math.inf, 1.0, 2.0, math.inf]
        top = [dict(zip(ps, _top_values(g["n"], *_edges(g, seed * 3 + i), ps, 1000))) for i, g in enumerate(graphs)]
        return _padded([k for _, _, k in requests], [top[g][p][:k] for g, p, k in requests])
    u, v, w = _edges(case, seed)
    if kind == "cliques":
        drawn = torch.ones(case["m"], dtype=torch.bool, device=DEV) if case["draws"] < 0 else \
            _drawn_edges(w, _ps(case)[0], case["draws"], int(seed))
        return *_padded([case["k"]], [_clique_values(case["n"], u, v, w, case["q"], _ps(case)[0], case["k"], drawn)]), None
    drawn = _drawn_edges(w, _ps(case)[0], case["draws"], int(seed)) if kind == "edges" else None
    vals = _top_values(case["n"], u, v, w, _ps(case), case["k"], drawn)
    if kind == "edges":
        return _padded([case["k"]], vals)
    if kind == "build" and case["where"] == "host":
        return [_padded([case["k"]], [x]) for x in vals]
    out = [torch.zeros(case["k"], dtype=torch.float64, device=DEV) for _ in vals]  # fewer than k: zeros follow
    for o, x in zip(out, vals):
        o[:x.numel()] = x
    return [(None, o, None) for o in out]
