"""The performance cases: the calls that a user of this package makes, over the sizes, degree laws
and options that they make them with.

Every input is a degree-corrected block model drawn on the GPU from the seed alone (the same recipe
as ``graphgen``: power-law degrees, rank-size communities, intra and inter stubs paired at random),
so that preparing a case takes a fraction of a second even at 100M edges.

    step      the scores of every node, then the top-K: one scoring step on a resident graph,
              launched directly or replayed from a captured step
    batch     the scores of many packed graphs (each with its own w_max)
    build     a pinned host CSR to the top-K list on the host: build with validation, score,
              top-K, copy, free
    removals  a resident graph is cloned, nodes and edges are removed, the rest is scored
    serve     a burst of what-if requests on resident graphs, to the last answer

``exact`` states the same values in 64 bits with plain torch: counts, weights, the Type-II sums and
the triangles of the cross-community subgraph, each straight from its definition.
"""
import math

import numpy as np
import torch

import paper_2508_01485_gb300 as rs

DEV = "cuda"

# Above these many candidate triples the 64-bit statement takes too long and is left out.
EXACT_CANDIDATES = 2_000_000_000


def _graph(n, k, size_min, gamma, dmin, dmax, mu):
    """The degree and community law of one graph."""
    return {"n": n, "k": k, "size_min": size_min, "gamma": gamma, "dmin": dmin, "dmax": dmax, "mu": mu}


def listed():
    return [
        # the 2,000-node block model of the tests: a small network scored once, where the launches
        # of a step are all that takes time
        {"name": "step_2k", "kind": "step", **_graph(2_000, 20, 100.0, 3.5, 7, 30, 0.1), "topk": 50, "mode": "direct", "option": ""},
        # a medium network scored again and again (a captured step replayed): the batch members'
        # and parity tests' shape, an odd size
        {"name": "step_33k_replay", "kind": "step", **_graph(33_333, 333, 50.0, 2.5, 8, 5000, 0.2), "topk": 100, "mode": "replay", "option": ""},
        # a larger one of the same law, launched directly
        {"name": "step_200k", "kind": "step", **_graph(200_001, 2_000, 50.0, 2.5, 7, 5000, 0.2), "topk": 100, "mode": "direct", "option": ""},
        # the strict reading of the triads, at a parity test's size
        {"name": "step_100k_strict", "kind": "step", **_graph(100_003, 1_000, 50.0, 2.5, 7, 1000, 0.2), "topk": 100, "mode": "direct", "option": "strict"},
        # 1M nodes, 1,000 communities, minimum degree 8: the mid-size benchmark
        {"name": "step_1m", "kind": "step", **_graph(1_000_000, 1_000, 50.0, 2.5, 8, 5000, 0.2), "topk": 1000, "mode": "direct", "option": ""},
        # the same with the literal minimum degree 2 and the top 1% of the nodes ranked, replayed
        {"name": "step_1m_dmin2", "kind": "step", **_graph(1_000_000, 1_000, 50.0, 2.5, 2, 5000, 0.2), "topk": 10_000, "mode": "replay", "option": ""},
        # hub-skewed: degrees to 100,000, heavy triangles, 12,500 communities
        {"name": "step_2m_hub", "kind": "step", **_graph(2_000_000, 12_500, 1.0, 2.1, 5, 100_000, 0.1), "topk": 1000, "mode": "direct", "option": ""},
        # the default benchmark: 8M nodes, 100M edges, 50,000 communities
        {"name": "step_8m_hub", "kind": "step", **_graph(8_000_000, 50_000, 1.0, 2.1, 5, 100_000, 0.1), "topk": 1000, "mode": "direct", "option": ""},
        # many independent graphs packed into one CSR, sizes log-uniform
        {"name": "batch_256", "kind": "batch", "graphs": 256, "n_min": 500, "n_max": 200_000, "gamma": 2.5, "dmin": 8, "dmax": 5000, "mu": 0.2},
        # a network arrives in host memory: everything from there to its ranking
        {"name": "build_1m", "kind": "build", **_graph(1_000_000, 1_000, 50.0, 2.5, 8, 5000, 0.2), "topk": 1000},
        # a robustness experiment's pass: the top nodes and some edges removed, the rest scored
        {"name": "removals_500k", "kind": "removals", **_graph(500_009, 500, 50.0, 2.5, 8, 5000, 0.2), "nodes": 5_000, "edges": 5_000},
        # a burst of concurrent what-if requests on resident networks of 10K to 1M nodes
        {"name": "serve_burst", "kind": "serve", "graphs": 4, "n_min": 10_000, "n_max": 1_000_000, "requests": 24, "slots": 8, "topk": 100},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _odd(rng, x):
    return x | 1 if rng.random() < 0.7 else x


def draw(rng):
    kind = rng.choice(["step", "step", "step", "hub", "hub", "batch", "build", "removals", "serve"])
    gamma, dmin, mu = round(rng.uniform(2.3, 3.0), 2), rng.randint(2, 9), round(rng.uniform(0.1, 0.4), 2)
    if kind == "step":
        n = _odd(rng, _log_uniform(rng, 1_500, 2_000_000))
        k = max(2, n // rng.choice([100, 300, 1000]))
        law = _graph(n, k, 50.0 if n >= 5_000 else 1.0, gamma, dmin, min(5000, n // 3), mu)
        option = rng.choice(["", "", "", "strict", "alg2", "reorder"])
        return {"kind": "step", **law, "topk": min(n, _log_uniform(rng, 10, 10_000)), "mode": rng.choice(["direct", "replay"]),
                "option": "" if option == "strict" and n > 300_000 else option}
    if kind == "hub":
        n = _odd(rng, _log_uniform(rng, 50_000, 4_000_000))
        law = _graph(n, max(2, n // 160), 1.0, round(rng.uniform(2.1, 2.3), 2), 5, min(100_000, n // 10), round(rng.uniform(0.08, 0.12), 3))
        return {"kind": "step", **law, "topk": min(n, _log_uniform(rng, 10, 10_000)), "mode": rng.choice(["direct", "replay"]), "option": ""}
    if kind == "batch":
        return {"kind": "batch", "graphs": _log_uniform(rng, 4, 256), "n_min": 500, "n_max": rng.choice([2_000, 20_000, 200_000]), "gamma": gamma,
                "dmin": dmin, "dmax": 5000, "mu": mu}
    if kind == "build":
        n = _odd(rng, _log_uniform(rng, 2_000, 2_000_000))
        return {"kind": "build", **_graph(n, max(2, n // rng.choice([100, 1000])), 20.0, gamma, dmin, min(5000, n // 3), mu), "topk": min(n, 1000)}
    if kind == "removals":
        n = _odd(rng, _log_uniform(rng, 10_000, 1_000_000))
        return {"kind": "removals", **_graph(n, max(2, n // rng.choice([100, 1000])), 50.0, gamma, max(4, dmin), min(5000, n // 3), mu),
                "nodes": _log_uniform(rng, 1, n // 50), "edges": _log_uniform(rng, 1, n // 50)}
    return {"kind": "serve", "graphs": rng.randint(1, 5), "n_min": 10_000, "n_max": _log_uniform(rng, 50_000, 1_000_000), "requests": rng.randint(1, 32),
            "slots": rng.choice([1, 4, 8, 16]), "topk": rng.choice([10, 100])}


# ---- inputs -----------------------------------------------------------------------------------


def _community_sizes(n, k, size_min):
    """Rank-size communities max(size_min, c / r), rounded to a total of n."""
    r = np.arange(1, k + 1, dtype=np.float64)
    size_min = min(size_min, n / k)
    lo, hi = 0.0, 2.0 * n
    for _ in range(100):
        c = 0.5 * (lo + hi)
        lo, hi = (lo, c) if np.maximum(c / r, size_min).sum() > n else (c, hi)
    s = np.maximum(hi / r, size_min)
    size = np.maximum(np.floor(s).astype(np.int64), 1)
    rest = int(n - size.sum())
    if rest > 0:
        size += np.bincount(np.argsort(size - s, kind="stable")[np.arange(rest) % k], minlength=k)
    while rest < 0:
        big = np.flatnonzero(size > 1)[-(-rest):]
        size[big] -= 1
        rest += len(big)
    return size


def _pairs(stubs, group, gen):
    """The stubs of each group paired at random (one is left over where their number is odd)."""
    key = (group << 31) + torch.randint(0, 1 << 31, stubs.shape, generator=gen, device=DEV)
    key, order = torch.sort(key, stable=True)
    group, stubs = key >> 31, stubs[order]
    count = torch.bincount(group)
    first = torch.cumsum(count, 0) - count
    at = torch.arange(stubs.numel(), device=DEV) - first[group]
    a = torch.nonzero((at % 2 == 0) & (at + 1 < count[group])).flatten()
    return stubs[a], stubs[a + 1]


def _draw_csr(parts, gen):
    """Graphs of the given laws side by side: offsets int64, cols int32 and labels int32, the
    labels distinct between graphs."""
    lab, gid, din, dout = [], [], [], []
    base = 0
    for i, p in enumerate(parts):
        size = torch.from_numpy(_community_sizes(p["n"], p["k"], p["size_min"])).to(DEV)
        c = torch.repeat_interleave(torch.arange(p["k"], device=DEV), size)[torch.randperm(p["n"], generator=gen, device=DEV)]
        d = torch.arange(p["dmin"], max(p["dmin"] + 1, min(p["dmax"], p["n"] - 1) + 1), dtype=torch.float64, device=DEV)
        cdf = torch.cumsum(d ** -p["gamma"], 0)
        u = torch.rand(p["n"], dtype=torch.float64, generator=gen, device=DEV) * cdf[-1]
        deg = p["dmin"] + torch.clamp(torch.searchsorted(cdf, u, right=True), max=d.numel() - 1)
        inner = torch.minimum(torch.floor((1.0 - p["mu"]) * deg + 0.5).to(torch.int64), size[c] - 1)
        lab.append(c + base)
        gid.append(torch.full_like(c, i))
        din.append(inner)
        dout.append(deg - inner)
        base += p["k"]
    lab, gid, din, dout = torch.cat(lab), torch.cat(gid), torch.cat(din), torch.cat(dout)
    n = lab.numel()
    node = torch.arange(n, device=DEV)
    s = torch.repeat_interleave(node, din)
    x, y = _pairs(s, lab[s], gen)
    keep = x != y
    es = [torch.minimum(x, y)[keep] * n + torch.maximum(x, y)[keep]]
    s = torch.repeat_interleave(node, dout)
    for _ in range(4):                       # pairs inside one community are paired again
        if s.numel() < 2:
            break
        x, y = _pairs(s, gid[s], gen)
        keep = lab[x] != lab[y]
        es.append(torch.minimum(x, y)[keep] * n + torch.maximum(x, y)[keep])
        s = torch.cat([x[~keep], y[~keep]])
    e = torch.unique(torch.cat(es))
    del s, x, y, keep, es
    u, v = e // n, e % n
    e = torch.sort(torch.cat([e, v * n + u])).values
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    offsets[1:] = torch.cumsum(torch.bincount(torch.div(e, n, rounding_mode="floor"), minlength=n), 0)
    return offsets, (e % n).to(torch.int32), lab.to(torch.int32)


def _sizes(case):
    """Node counts of a batch's or a server's graphs: even on a logarithmic scale, odd sizes."""
    g = case["graphs"]
    at = [(i + 0.5) / g for i in range(g)] if case["kind"] == "batch" else [i / max(1, g - 1) if g > 1 else 1.0 for i in range(g)]
    return [int(round(case["n_min"] * (case["n_max"] / case["n_min"]) ** a)) for a in at]


def _laws(case):
    if case["kind"] == "batch":
        return [_graph(n, max(2, n // 100), 50.0 if n >= 5000 else 1.0, case["gamma"], case["dmin"], case["dmax"], case["mu"]) for n in _sizes(case)]
    if case["kind"] == "serve":
        return [_graph(n, max(2, n // 1000), 50.0, 2.5, 8, 5000, 0.2) for n in _sizes(case)]
    return [{k: case[k] for k in ("n", "k", "size_min", "gamma", "dmin", "dmax", "mu")}]


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _removal_lists(offsets, cols, rng, nodes, edges, hot):
    """Node ids and edges to remove: a share `hot` of the targets among the 1% of largest degree."""
    deg = np.diff(offsets)
    n = len(deg)
    top = np.argsort(-deg, kind="stable")[: max(1, n // 100)]
    pick = lambda m: np.where(rng.random(m) < hot, top[rng.integers(0, len(top), m)], rng.integers(0, n, m))  # noqa: E731
    nd = np.unique(pick(nodes)).astype(np.int32) if nodes else np.zeros(0, np.int32)
    src = pick(edges)
    src = src[deg[src] > 0]
    dst = cols[offsets[src] + (rng.random(len(src)) * deg[src]).astype(np.int64)]
    return nd, np.stack([src, dst], 1).astype(np.int32)


def _requests(case, graphs, seed):
    """The burst: a graph uniformly, a removal count log-uniform on [1, 10000] (at most a tenth of
    the nodes), half of the requests nodes and half edges, 70% of the targets well connected."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["requests"]):
        gi = int(rng.integers(0, len(graphs)))
        off, cols = graphs[gi]
        n = len(off) - 1
        # counts at even steps of the logarithm, so that bursts of other seeds cost alike
        m = int(min(round(10000.0 ** ((i + 0.5) / case["requests"])), max(1, n // 10)))
        nd, ed = _removal_lists(off, cols, rng, m if i % 2 else 0, 0 if i % 2 else m, 0.7)
        out.append((gi, nd, ed))
    return out


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "serve":
        host, graphs = [], []
        for law in _laws(case):
            off, cols, lab = _draw_csr([law], gen)
            graphs.append(rs.Graph.build(off, cols, lab, law["k"], validate=False))
            host.append((off.cpu().numpy(), cols.cpu().numpy()))
        st["server"] = rs.Server(graphs, max_slots=case["slots"], budget_bytes=32 << 30, max_top_k=case["topk"])
        st["requests"] = _requests(case, host, seed)
        st["topk"] = case["topk"]
        return st
    laws = _laws(case)
    off, cols, lab = _draw_csr(laws, gen)
    n = lab.numel()
    st["scores"] = torch.empty(n, dtype=torch.float64, device=DEV)
    if kind == "batch":
        gno = np.concatenate([[0], np.cumsum([p["n"] for p in laws])]).astype(np.int64)
        gk = np.array([p["k"] for p in laws], np.int32)
        first = np.repeat(np.concatenate([[0], np.cumsum(gk)[:-1]]), np.diff(gno)).astype(np.int32)
        st["graph"] = rs.Graph.build_batch(gno, gk, off.cpu().numpy(), cols.cpu().numpy(), lab.cpu().numpy() - first, validate=False)
        return st
    k = case["k"]
    if kind == "build":
        st["host"] = [t.cpu().pin_memory() for t in (off, cols, lab)]
        st["arrays"] = [t.numpy() for t in st["host"]]
        st["k"] = k
    else:
        opt = case.get("option", "")
        st["graph"] = rs.Graph.build(off, cols, lab, k, validate=False, alg2=opt == "alg2", strict=opt == "strict", reorder=opt == "reorder")
    if kind == "removals":
        st["nodes"], st["edges"] = _removal_lists(off.cpu().numpy(), cols.cpu().numpy(), np.random.default_rng(seed), case["nodes"], case["edges"], 0.7)
        return st
    st["topk"] = case["topk"]
    st["ids"] = torch.empty(case["topk"], dtype=torch.int32, device=DEV)
    st["vals"] = torch.empty(case["topk"], dtype=torch.float64, device=DEV)
    if case.get("mode") == "replay":
        st["step"] = st["graph"].capture_step(st["scores"], case["topk"], st["ids"], st["vals"])
    return st


# ---- one pass ---------------------------------------------------------------------------------


def run(st):
    kind = st["kind"]
    if kind == "step":
        if "step" in st:
            st["step"].launch()
        else:
            st["graph"].score_into(st["scores"])
            st["graph"].topk_into(st["scores"], st["topk"], st["ids"], st["vals"])
        return {"scores": st["scores"], "ids": st["ids"], "vals": st["vals"]}
    if kind == "batch":
        return {"scores": st["graph"].score_into(st["scores"])}
    if kind == "build":
        g = rs.Graph.build(*st["arrays"], st["k"], validate=True)
        g.score_into(st["scores"])
        g.topk_into(st["scores"], st["topk"], st["ids"], st["vals"])
        ids, vals = st["ids"].cpu(), st["vals"].cpu()
        g.close()
        return {"scores": st["scores"], "ids": ids, "vals": vals}
    if kind == "removals":
        g = st["graph"].clone()
        applied = g.apply_removals(st["nodes"], st["edges"])
        g.score_into(st["scores"])
        g.close()
        return {"scores": st["scores"], "applied": applied}
    srv, k = st["server"], st["topk"]
    order = {}
    for i, (gi, nd, ed) in enumerate(st["requests"]):
        order[srv.submit(gi, nd, ed, top_k=k)] = i
    ids = np.zeros((len(order), k), np.int32)
    vals = np.zeros((len(order), k), np.float64)
    status = np.zeros(len(order), np.int32)
    left = len(order)
    while left:
        for t, s, _, i, v in srv.poll(block=True):
            at = order[t]
            ids[at], vals[at], status[at] = i, v, s
            left -= 1
    return {"ids": ids, "vals": vals, "status": status}


def _mean_degree(p):
    d = np.arange(p["dmin"], max(p["dmin"] + 1, min(p["dmax"], p["n"] - 1) + 1), dtype=np.float64)
    w = d ** -p["gamma"]
    return float((d * w).sum() / w.sum())


def _csr_bytes(p):
    """Offsets, columns and labels of one graph (the degree law's mean)."""
    return 8 * (p["n"] + 1) + 4 * p["n"] * _mean_degree(p) + 4 * p["n"]


def work(case):
    """The CSR read once and every score written once (the triangles, which depend on the draw, are
    not counted); per CSR entry a count, per node the dozen operations of its weight and score."""
    laws = _laws(case)
    nodes = sum(p["n"] for p in laws)
    entries = sum(p["n"] * _mean_degree(p) for p in laws)
    kind = case["kind"]
    if kind == "serve":                      # every answer ranks its changed graph's scores
        return {"bytes": case["requests"] * (16 * nodes / len(laws) + 12 * case["topk"]), "flops": case["requests"] * 2 * nodes / len(laws)}
    return {"bytes": sum(map(_csr_bytes, laws)) + 8 * nodes + 12 * case.get("topk", 0), "flops": entries + 12 * nodes}


# ---- the same values in 64 bits ---------------------------------------------------------------


def _ranges(first, count):
    """For every i: first[i], first[i] + 1, .. first[i] + count[i] - 1; and the i of each."""
    i = torch.repeat_interleave(torch.arange(count.numel(), device=DEV), count)
    at = torch.cumsum(count, 0) - count
    return first[i] + (torch.arange(i.numel(), device=DEV) - at[i]), i


def _chunks(count, most=1 << 25):
    """Cuts [0, len(count)) into runs of about `most` in all."""
    total = torch.cumsum(count, 0)
    cuts, at, n = [], 0, count.numel()
    while at < n:
        done = int(total[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(total, done + most)))
        cuts.append((at, min(to, n)))
        at = min(to, n)
    return cuts


def _find(keys, q):
    """Positions of q in the ascending keys (-1 where it is not there)."""
    at = torch.clamp(torch.searchsorted(keys, q), max=max(0, keys.numel() - 1))
    return torch.where(keys[at] == q, at, torch.full_like(at, -1))


def _exact_scores(off, cols, lab, graph_of, ks, option=""):
    """R(u) of every node of the graphs packed side by side (labels distinct between graphs), or
    None where there are too many candidate triangles."""
    n, K = lab.numel(), int(sum(ks))
    deg = off[1:] - off[:-1]
    u = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    v = cols.to(torch.int64)
    lab = lab.to(torch.int64)
    # counts f_v(c), one entry per (node, neighbour community)
    pairs, which, f = torch.unique(u * K + lab[v], return_inverse=True, return_counts=True)
    pn = torch.div(pairs, K, rounding_mode="floor")
    f = f.to(torch.float64)
    flogf = f * torch.log2(f)
    X = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, pn, flogf)
    L = torch.bincount(pn, minlength=n).to(torch.float64)
    T = deg.to(torch.float64)

    def weight(Y, Xr, size):
        h = torch.log2(torch.clamp(Y, min=1.0)) - Xr / torch.clamp(Y, min=1.0)
        return torch.where(size > 1, torch.clamp(h, min=0.0) * size, torch.zeros_like(h))

    w = weight(T[pn] - f, X[pn] - flogf, L[pn] - 1)
    w0 = weight(T, X, L - 1 if option == "alg2" else L)   # a community absent from N(v)
    kn = torch.tensor(ks, dtype=torch.float64, device=DEV)[graph_of]
    wmax = torch.zeros(len(ks), dtype=torch.float64, device=DEV)
    wmax.scatter_reduce_(0, graph_of[pn], w, "amax")
    wmax.scatter_reduce_(0, graph_of, torch.where(L < kn, w0, torch.zeros_like(w0)), "amax")
    sig, own = w ** (1 / 3), (pairs % K) == lab[pn]
    s = w0 ** (1 / 3)
    s[pn[own]] = sig[own]
    # Type-II: sigma_w(C(u))^2 (Q_w(C(u)) - s_u) from every w to its neighbours u elsewhere
    Q = torch.zeros_like(f).index_add_(0, which, s[v])
    members = f[which]
    cross = lab[u] != lab[v]
    push = torch.where(members > 1, sig[which] ** 2 * (Q[which] - s[v]), torch.zeros(1, dtype=torch.float64, device=DEV))
    acc = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, v[cross], push[cross])
    # the cross-community subgraph: entry (a, b) carries S(a -> b) = sigma_a(C(b))
    a, b, S = u[cross], v[cross], sig[which][cross]
    key = a * n + b
    R = S[_find(key, b * n + a)]
    dx = torch.bincount(a, minlength=n)
    if option == "strict":
        # a closed triangle (u, w, v) with C(v) = C(u) is no triad: taken out of the Type-II sums
        inner = ~cross & (u < v)
        p, q = u[inner], v[inner]
        p, q = torch.where(dx[p] <= dx[q], p, q), torch.where(dx[p] <= dx[q], q, p)
        start = torch.cumsum(dx, 0) - dx
        if int(dx[p].sum()) > EXACT_CANDIDATES:
            return None
        for lo, hi in _chunks(dx[p]):
            e, i = _ranges(start[p[lo:hi]], dx[p[lo:hi]])
            o = _find(key, q[lo:hi][i] * n + b[e])
            e, i, o = e[o >= 0], i[o >= 0], o[o >= 0]
            x, y = p[lo:hi][i], q[lo:hi][i]
            acc.index_add_(0, x, -R[e] ** 2 * s[y])
            acc.index_add_(0, y, -R[e] ** 2 * s[x])
    # Type-I: its triangles, each once, edges pointing to the higher (dx, id)
    up = (dx[b] > dx[a]) | ((dx[b] == dx[a]) & (b > a))
    a, b, S, R = a[up], b[up], S[up], R[up]
    key = key[up]
    od = torch.bincount(a, minlength=n)
    start = torch.cumsum(od, 0) - od
    short = torch.where(od[a] <= od[b], a, b)
    cand = od[short]
    if int(cand.sum()) > EXACT_CANDIDATES:
        return None
    for lo, hi in _chunks(cand):
        e, i = _ranges(start[short[lo:hi]], cand[lo:hi])
        i += lo
        o = _find(key, (a[i] + b[i] - short[i]) * n + b[e])
        hit = o >= 0
        e, i, o = e[hit], i[hit], o[hit]
        from_a = short[i] == a[i]
        ac, bc, ab = torch.where(from_a, e, o), torch.where(from_a, o, e), i
        c = b[ac]
        # S(x -> y): S along an edge, R against it
        acc.index_add_(0, a[ab], R[ab] * R[ac] * (S[bc] + R[bc]))
        acc.index_add_(0, b[ab], S[ab] * R[bc] * (S[ac] + R[ac]))
        acc.index_add_(0, c, S[ac] * S[bc] * (S[ab] + R[ab]))
    top = wmax[graph_of]
    denom = top * T * (T - 1)
    return torch.where((T >= 2) & (top > 0), acc / torch.where(denom > 0, denom, torch.ones_like(denom)), torch.zeros_like(acc))


def _without(off, cols, nodes, edges):
    """The CSR without the nodes' edges and the edges, and how many of them were there."""
    n = off.numel() - 1
    u = torch.repeat_interleave(torch.arange(n, device=DEV), off[1:] - off[:-1])
    v = cols.to(torch.int64)
    gone = torch.zeros(n, dtype=torch.bool, device=DEV)
    nd = torch.from_numpy(np.asarray(nodes, np.int64).reshape(-1)).to(DEV)
    gone[nd] = True
    keep = ~(gone[u] | gone[v])
    u, v = u[keep], v[keep]
    e = torch.from_numpy(np.asarray(edges, np.int64).reshape(-1, 2)).to(DEV)
    x = torch.cat([e[:, 0] * n + e[:, 1], e[:, 1] * n + e[:, 0]])
    keep = ~torch.isin(u * n + v, x)
    u, v = u[keep], v[keep]
    out = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    out[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return out, v.to(torch.int32)


def _best(scores, k):
    return torch.sort(scores, descending=True).values[:k]


def exact(case, seed):
    gen = _generator(seed)
    laws = _laws(case)
    if case["kind"] == "serve":
        graphs = [_draw_csr([p], gen) for p in laws]
        vals = []
        for gi, nd, ed in _requests(case, [(o.cpu().numpy(), c.cpu().numpy()) for o, c, _ in graphs], seed):
            off, cols, lab = graphs[gi]
            o, c = _without(off, cols, nd, ed)
            one = torch.zeros(lab.numel(), dtype=torch.int64, device=DEV)
            vals.append(_best(_exact_scores(o, c, lab, one, [laws[gi]["k"]]), case["topk"]))
        return {"ids": None, "vals": torch.stack(vals), "status": None}
    off, cols, lab = _draw_csr(laws, gen)
    if case["kind"] == "removals":
        nd, ed = _removal_lists(off.cpu().numpy(), cols.cpu().numpy(), np.random.default_rng(seed), case["nodes"], case["edges"], 0.7)
        off, cols = _without(off, cols, nd, ed)
    graph_of = torch.repeat_interleave(torch.arange(len(laws), device=DEV), torch.tensor([p["n"] for p in laws], device=DEV))
    scores = _exact_scores(off, cols, lab, graph_of, [p["k"] for p in laws], case.get("option", ""))
    if scores is None:
        return None
    if case["kind"] == "batch":
        return {"scores": scores}
    if case["kind"] == "removals":
        return {"scores": scores, "applied": None}
    return {"scores": scores, "ids": None, "vals": _best(scores, case["topk"])}
