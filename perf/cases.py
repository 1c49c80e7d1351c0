"""The calls this library is measured on: plain descriptions of a graph, a
sketch and a call, the inputs a program has in hand before it, and the call
itself through the public entry points.

Kinds of call:
  query   skis_estimate: a batch of seed sets against a resident sketch
  serve   the continuous-batching server: a burst of requests, submitted,
          driven and polled
  sample  a new sketch of a loaded graph, its samples, and the greedy seeds
  load    a graph load; small graphs are exported whole, larger ones are put
          to their first use (a pilot sketch, its seeds and a query batch)
  step    load, samples, greedy and a query batch in one: a whole run
  dssa    influence maximisation by doubling sketches

Graphs are drawn on the GPU with torch: Erdos-Renyi ("er"), Chung-Lu with a
power-law degree exponent ("chunglu") and R-MAT ("rmat").
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1709_03565_gb300 as skis

SKETCH_SEED = 0x5EED


def _case(kind, graph, n, m, model, **kw):
    c = dict(kind=kind, graph=graph, n=n, m=m, model=model, beta=2.1, samples=0, first_step="rejection",
             sampler="iis", k=0, queries=0, size_lo=10, size_hi=10, space="device", split="default")
    c.update(kw)
    return c


def listed():
    return [
        # one influence query of a small resident sketch, as an interactive program asks it: the smallest call,
        # all latency (the Erdos-Renyi configuration: n = 10,000, m = 100,000, 100,000 samples, sets of 10)
        dict(_case("query", "er", 10_000, 100_000, "wc", samples=100_000, queries=1, space="host"),
             name="query-er-1"),
        # a batch of 64 queries against a large sketch with no index built: a scan of its members
        dict(_case("query", "chunglu", 1_000_000, 10_000_000, "tri", samples=10_000_000, first_step="bucket",
                   queries=64), name="query-chunglu-scan-64"),
        # the query service at saturation: a burst of requests of uneven size (Chung-Lu 4M / 70M)
        dict(_case("serve", "chunglu", 4_000_000, 70_000_000, "wc", samples=5_000_000, queries=1024, size_lo=1,
                   size_hi=1000, space="host"), name="serve-chunglu-1024"),
        # a small influence-maximisation run on a loaded graph: launches and host round trips count
        dict(_case("sample", "er", 10_000, 100_000, "wc", samples=100_000, k=10), name="sample-er-wc"),
        # the same at the size of the trivalency configuration: short samples, ten million of them
        dict(_case("sample", "chunglu", 1_000_000, 10_000_000, "tri", samples=10_000_000, first_step="bucket", k=50),
             name="sample-chunglu-tri"),
        # many seeds from a weighted-cascade sketch: the greedy rounds are most of the call
        dict(_case("sample", "chunglu", 1_000_000, 17_500_000, "wc", samples=1_000_000, k=1000),
             name="sample-chunglu-wc-k1000"),
        # the Linear Threshold model: random walks instead of a BFS
        dict(_case("sample", "chunglu", 1_000_000, 10_000_000, "lt", samples=2_000_000, k=50),
             name="sample-chunglu-lt"),
        # samples that reach the hubs of an R-MAT graph, hundreds of thousands of coins each
        dict(_case("sample", "rmat", 1 << 22, 1 << 27, "wc", samples=200_000, first_step="bucket", k=100,
                   split="heavy"), name="sample-rmat-wc"),
        # a small graph loaded from host arrays and read back whole (an odd edge count)
        dict(_case("load", "er", 10_000, 100_003, "wc", space="host"), name="load-er"),
        # a serving graph loaded from device arrays, and its first use
        dict(_case("load", "chunglu", 4_000_000, 70_000_000, "wc", samples=1 << 16, k=10, queries=64),
             name="load-chunglu-70m"),
        # a whole run on explicit trivalency probabilities, sizes off every power of two
        dict(_case("step", "chunglu", 333_331, 3_000_017, "tri", samples=1_500_007, first_step="bucket", k=50,
                   queries=100, size_lo=1, size_hi=100), name="step-chunglu-tri"),
        # influence maximisation with a guarantee (DSSA-style doubling), a tenth of the 40M / 1.4B configuration
        dict(_case("dssa", "chunglu", 4_000_000, 140_000_000, "wc", beta=2.0, k=100), name="dssa-chunglu"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "serve", "sample", "sample", "sample", "load", "step", "dssa"])
    if kind == "dssa":
        n = _logint(rng, 100_000, 2_000_000)
        return _case(kind, "chunglu", n, n * rng.randint(10, 30) + rng.randint(0, 3), "wc",
                     beta=rng.choice([2.0, 2.1]), k=_logint(rng, 1, 100))
    graph = rng.choice(["er", "chunglu", "chunglu", "rmat"] if kind in ("sample", "step", "load") else
                       ["er", "chunglu", "chunglu"])
    first_step = rng.choice(["rejection", "bucket"])
    sampler = rng.choice(["iis", "iis", "iis", "ris"])
    split = "default"
    if graph == "er":
        n = _logint(rng, 1_000, 50_000)
        m = n * rng.randint(4, 12) + rng.randint(0, 3)
        model = rng.choice(["wc", "wc", "tri", "lt"])
        samples = _logint(rng, 10_000, 400_000)
    elif graph == "chunglu":
        n = _logint(rng, 50_000, 2_000_000)
        m = n * rng.randint(6, 18) + rng.randint(0, 3)
        model = rng.choice(["wc", "tri", "tri", "lt"])
        samples = _logint(rng, 50_000, 10_000_000 if model == "tri" else 1_000_000)
    else:
        scale = rng.randint(16, 22)
        n = 1 << scale
        m = 32 * n + rng.randint(0, 3)
        model = "wc"
        samples = _logint(rng, 2_000, 150_000)
        split = rng.choice(["default", "heavy"])
    if model == "lt":
        first_step = "rejection"
    kw = dict(samples=samples, first_step=first_step, sampler=sampler, split=split)
    if kind == "query":
        kw.update(queries=_logint(rng, 1, 256), size_lo=1, size_hi=_logint(rng, 1, 300),
                  space=rng.choice(["host", "device"]))
    elif kind == "serve":
        kw.update(queries=_logint(rng, 16, 1024), size_lo=1, size_hi=_logint(rng, 1, 1000), space="host")
    elif kind == "sample":
        kw.update(k=_logint(rng, 1, 1000))
    elif kind == "load":
        kw = dict(space=rng.choice(["host", "device"]))
        if n * m > 10**10:
            kw = dict(samples=1 << 14, k=10, queries=64, split=split)
    else:
        kw.update(k=_logint(rng, 1, 200), queries=64, size_lo=1, size_hi=100)
    return _case(kind, graph, n, m, model, **kw)


# ------------------------------------------------------------------ inputs
def _weight_sum(n, i0, ex):
    head = min(n, 65536)
    tot = float(((np.arange(head) + i0 + 1.0) ** ex).sum())
    if head < n:
        a, b = head - 0.5 + i0 + 1.0, n - 0.5 + i0 + 1.0
        tot += (math.log(b / a) if ex == -1.0 else (b ** (ex + 1.0) - a ** (ex + 1.0)) / (ex + 1.0))
    return tot


def _edges(case, seed):
    """Edge arrays (int32, CUDA) of the case's graph; self-loops are shifted away, parallel edges kept."""
    n, m = case["n"], case["m"]
    g = torch.Generator(device="cuda").manual_seed(0x9E37 + 7919 * int(seed))
    if case["graph"] == "er":
        src = torch.randint(0, n, (m,), generator=g, device="cuda")
        dst = (src + 1 + torch.randint(0, n - 1, (m,), generator=g, device="cuda")) % n
    elif case["graph"] == "chunglu":
        # expected degree of rank i proportional to (i + i0 + 1)^(-1/(beta - 1)), the largest sqrt(m);
        # out- and in-weights attached to the vertices by two independent permutations
        ex = -1.0 / (case["beta"] - 1.0)
        lo, hi = 0.0, float(n)
        for _ in range(60):
            i0 = 0.5 * (lo + hi)
            if m * (i0 + 1.0) ** ex / _weight_sum(n, i0, ex) > math.sqrt(m):
                lo = i0
            else:
                hi = i0
        cdf = np.cumsum((np.arange(n) + hi + 1.0) ** ex)  # on the host: a float scan on the GPU varies in its last bits
        cdf = torch.from_numpy(cdf / cdf[-1]).cuda()
        ends = []
        for _ in range(2):
            perm = torch.randperm(n, generator=g, device="cuda")
            u = torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
            ends.append(perm[torch.searchsorted(cdf, u).clamp_(max=n - 1)])
        src, dst = ends
        dst = torch.where(src == dst, (dst + 1) % n, dst)
    else:
        a, b, c = 0.57, 0.19, 0.19
        src = torch.zeros(m, dtype=torch.int32, device="cuda")
        dst = torch.zeros(m, dtype=torch.int32, device="cuda")
        for _ in range(n.bit_length() - 1):
            x = torch.rand(m, generator=g, device="cuda")
            src.mul_(2).add_(x >= a + b)
            dst.mul_(2).add_(((x >= a) & (x < a + b)) | (x >= a + b + c))
        dst = torch.where(src == dst, (dst + 1) % n, dst)
    src, dst = src.to(torch.int32), dst.to(torch.int32)
    p = None
    if case["model"] == "tri":
        levels = torch.tensor([0.1, 0.01, 0.001], dtype=torch.float64, device="cuda")
        p = levels[torch.randint(0, 3, (m,), generator=g, device="cuda")]
    if case["space"] == "host" and case["kind"] == "load":
        src, dst, p = src.cpu().numpy(), dst.cpu().numpy(), None if p is None else p.cpu().numpy()
    return src, dst, p


def _queries(case, seed):
    """Seed sets (offsets int64, seeds int32, numpy): sizes log-uniform, members distinct and uniform."""
    rng = np.random.default_rng([11, int(seed)])
    q, lo, hi = case["queries"], case["size_lo"], min(case["size_hi"], case["n"])
    sizes = np.clip(np.floor(np.exp(rng.uniform(math.log(lo), math.log(hi + 1), q))), lo, hi).astype(np.int64)
    off = np.zeros(q + 1, np.int64)
    np.cumsum(sizes, out=off[1:])
    seeds = [rng.choice(case["n"], int(x), replace=False, shuffle=False) for x in sizes]
    return off, np.concatenate(seeds).astype(np.int32)


def _load(case, edges):
    src, dst, p = edges
    if case["model"] == "lt":
        return skis.skis_load_graph_lt(case["n"], src, dst, None, skis.SKIS_W_WC)
    if case["model"] == "tri":
        return skis.skis_load_graph(case["n"], src, dst, p, skis.SKIS_W_EXPLICIT_P)
    return skis.skis_load_graph(case["n"], src, dst, None, skis.SKIS_W_WC)


def _sketch(case, graph):
    s = skis.skis_sketch_create(graph, SKETCH_SEED)
    if case["first_step"] == "bucket" and case["model"] != "lt":
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_FIRST_STEP, 1)
    if case["sampler"] == "ris":
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_SAMPLER, 1)
    if case["split"] == "heavy":  # the split the autotuner picks where nearly every sample reaches a hub
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_THREAD_MAX_DEG, 0)
        skis.skis_sketch_set_option(s, skis.SKIS_OPT_WARP_MAX_COINS, 4096)
    skis.skis_sample(s, case["samples"])
    return s


def prepare(case, seed):
    edges = _edges(case, seed)
    st = dict(case=case)
    if case["queries"]:
        off, seeds = _queries(case, seed)
        if case["kind"] == "serve":
            st["requests"] = [seeds[off[b]:off[b + 1]] for b in range(case["queries"])]
        elif case["space"] == "device":
            st["off"], st["seeds"] = torch.from_numpy(off).cuda(), torch.from_numpy(seeds).cuda()
        else:
            st["off"], st["seeds"] = off, seeds
    if case["kind"] in ("load", "step"):
        st["edges"] = edges
        return st
    st["graph"] = _load(case, edges)
    if case["kind"] in ("query", "serve"):
        st["sketch"] = _sketch(case, st["graph"])
    if case["kind"] == "serve":
        st["server"] = skis.skis_server_create(st["sketch"], slots=4, max_batch=64, seed_capacity=1 << 16)
    return st


# -------------------------------------------------------------------- runs
def _estimate(s, off, seeds):
    if isinstance(off, np.ndarray):
        return skis.skis_estimate(s, off, seeds)
    q = off.numel() - 1
    cov = torch.empty(q, dtype=torch.int64, device=off.device)
    est = torch.empty(q, dtype=torch.float64, device=off.device)
    return skis.skis_estimate(s, off, seeds, cov, est)


def _serve(server, requests):
    tickets = []
    left = len(requests)
    for i, seeds in enumerate(requests):
        tickets.append(skis.skis_server_submit(server, seeds))
        if i % 64 == 63:
            left -= len(skis.skis_server_progress(server))
    while left > 0:
        left -= len(skis.skis_server_progress(server, wait=True))
    answers = [skis.skis_server_poll(server, t) for t in tickets]
    return (np.array([x[0] for x in answers]), np.array([x[1] for x in answers]), np.array([x[2] for x in answers]))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "query":
        return _estimate(state["sketch"], state["off"], state["seeds"])
    if kind == "serve":
        return _serve(state["server"], state["requests"])
    if kind == "sample":
        s = _sketch(case, state["graph"])
        out = skis.skis_greedy_maxcover(s, case["k"])
        s.close()
        return out
    if kind == "dssa":
        seeds, res = skis.skis_dssa_maxinf(state["graph"], SKETCH_SEED + 4, SKETCH_SEED + 5, case["k"], 0.1,
                                           1.0 / case["n"], 0, 1 << 16, 1 << 26)
        return seeds, res
    g = _load(case, state["edges"])
    out = [skis.skis_graph_get_info(g)]
    if case["samples"] == 0:
        out.append(skis.skis_graph_export(g))
    else:
        s = _sketch(case, g)
        out.extend(skis.skis_greedy_maxcover(s, case["k"]))
        out.extend(_estimate(s, state["off"], state["seeds"]))
        if kind == "step":
            stats = skis.skis_sketch_stats(s)
            out.append({k: stats[k] for k in ("T", "entries", "coins", "retries")})
        s.close()
    g.close()
    return out


# ------------------------------------------------------------ floor of work
def _members(case):
    """Members of a sample, about: what the listed graphs give (for the floor of the bytes only)."""
    if case["sampler"] == "ris":
        return 2.0 if case["model"] == "tri" else 12.0
    return {"tri": 4.2, "lt": 18.0, "wc": 60.0 if case["graph"] == "er" else 70.0}[case["model"]]


def work(case):
    n, m, T = case["n"], case["m"], case["samples"]
    per_edge = 16 if case["model"] == "tri" else 8
    seeds = case["queries"] * math.sqrt(case["size_lo"] * case["size_hi"])
    entries = T * _members(case)
    answers = 16 * case["queries"] + 4 * seeds
    if case["kind"] == "query":  # every member of the sketch once
        return {"bytes": 4 * entries + answers, "flops": 0}
    if case["kind"] == "serve":  # the sample lists of the seeds
        return {"bytes": 4 * seeds * entries / n + answers, "flops": 0}
    if case["kind"] == "dssa":  # two sketches of some 2^17 samples each, grown and read
        T = 1 << 18
        entries = T * _members(case)
    # samples: headers (28 bytes) and members written, the members read once to choose seeds; the graph's
    # row and alias records of the sources
    sketch = T * (28 + 32) + 8 * entries + 20 * case["k"]
    if case["kind"] in ("sample", "dssa"):
        return {"bytes": sketch, "flops": 0}
    # load: edges (and probabilities) read, CSR, row, weight and alias records written
    load = m * per_edge + m * (16 if case["model"] == "tri" else 12) + n * 48
    return {"bytes": load + (sketch + 4 * entries + answers if T else 0), "flops": 0}


# ----------------------------------------------------------- exact results
# Erdos-Renyi graphs under weighted cascade with the rejection first step, from the definitions, in torch
# int64 and Python integers: small enough to be done again here. Larger sketches would take minutes.
_M32 = 0xFFFFFFFF
_DOM_SRC, _DOM_FIRST, _DOM_BFS = 1, 2, 3


def _hi32(x):
    return (x >> 32) & _M32


def _philox(q, retry, dom, j):
    """The four coin words of edge quads q of samples j: Philox4x32-10, key SKETCH_SEED."""
    x = [q & _M32, ((retry & 0xFFFFFF) << 4 | dom << 28) + torch.zeros_like(q), j & _M32, _hi32(j)]
    k0, k1 = SKETCH_SEED & _M32, SKETCH_SEED >> 32
    for _ in range(10):
        pa, pb = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [_hi32(pb) ^ x[1] ^ k0, pb & _M32, _hi32(pa) ^ x[3] ^ k1, pa & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return torch.stack(x, -1)


def _mulhi64(hi, lo, b):
    """floor((hi 2^32 + lo) b / 2^64) for b < 2^62."""
    bh, bl = b >> 32, b & _M32
    mid = lo * bh + _hi32(lo * bl)
    mid2 = hi * bl + (mid & _M32)
    return hi * bh + (mid >> 32) + _hi32(mid2)


def _exact_graph(n, src, dst):
    """off, csr sources, thresholds per row, w, W, alias table (prob as Python integers' int64, alias)."""
    src, dst = src.long(), dst.long()
    key, _ = torch.sort(dst * n + src, stable=True)
    csr = key % n
    deg = torch.bincount(key // n, minlength=n)
    off = torch.zeros(n + 1, dtype=torch.int64, device=src.device)
    off[1:] = torch.cumsum(deg, 0)
    tau = torch.where(deg > 1, (1 << 32) // deg.clamp(min=1), torch.zeros_like(deg))
    tau[deg == 1] = 1 << 32
    c = (1 << 32) - tau
    Q = torch.full_like(deg, 1 << 62)
    for i in range(int(deg.max())):
        nxt = (Q >> 32) * c + _hi32((Q & _M32) * c)
        Q = torch.where(i < deg, nxt, Q)
    bits = (n - 1).bit_length()
    w = ((1 << 62) - Q) >> (bits + 1)
    W = int(w.sum())
    mass = [int(x) * n for x in w.tolist()]
    light, heavy = [v for v in range(n) if mass[v] < W], [v for v in range(n) if mass[v] >= W]
    prob, alias = [W] * n, list(range(n))
    h, excess, deficit = 0, mass[heavy[0]] - W, 0  # running sums: heavy excesses through h, light deficits so far
    for v in light:
        while excess < deficit:  # the first heavy item whose running excess covers the deficits before v
            prob[heavy[h]], alias[heavy[h]] = W + excess - deficit, heavy[h + 1]
            h += 1
            excess += mass[heavy[h]] - W
        prob[v], alias[v] = mass[v], heavy[h]
        deficit += W - mass[v]
    while h + 1 < len(heavy) and W + excess - deficit < W:
        prob[heavy[h]], alias[heavy[h]] = W + excess - deficit, heavy[h + 1]
        h += 1
        excess += mass[heavy[h]] - W
    dev = src.device
    return (off, csr, tau, w, W, 61 - bits, torch.tensor(prob, device=dev), torch.tensor(alias, device=dev))


def _live(off, csr, tau, j, v, retry, dom):
    """Live in-edges of the vertices v of samples j: (index into j, source)."""
    deg = off[v + 1] - off[v]
    row = torch.repeat_interleave(torch.arange(v.numel(), device=v.device), deg)
    e = off[v][row] + torch.arange(row.numel(), device=v.device) - (torch.cumsum(deg, 0) - deg)[row]
    x = _philox(e >> 2, retry, dom, j[row]).gather(1, (e & 3).unsqueeze(1)).squeeze(1)
    hit = x < tau[v][row]
    return row[hit], csr[e[hit]]


def _exact_sketch(case, off, csr, tau, W, prob, alias):
    """(sample, vertex) membership pairs of the case's sketch, sorted."""
    n, T = case["n"], case["samples"]
    j = torch.arange(T, device=off.device)
    x = _philox(torch.zeros_like(j), 0, _DOM_SRC, j)
    col = _mulhi64(x[:, 1], x[:, 0], n)
    v = torch.where(_mulhi64(x[:, 3], x[:, 2], W) < prob[col], col, alias[col])
    members, front = [j * n + v], []
    r = 0
    while j.numel():  # the conditioned first step: rounds until a coin is live
        row, u = _live(off, csr, tau, j, v, r, _DOM_FIRST)
        front.append(j[row] * n + u)
        wait = torch.ones_like(j, dtype=torch.bool)
        wait[row] = False
        j, v, r = j[wait], v[wait], r + 1
    seen, front = members[0], torch.unique(torch.cat(front))
    while True:
        front = front[~torch.isin(front, seen)]
        if front.numel() == 0:
            return torch.sort(seen)[0]
        seen = torch.cat([seen, front])
        j, v = front // n, front % n
        row, u = _live(off, csr, tau, j, v, 0, _DOM_BFS)
        front = torch.unique(j[row] * n + u)


def exact(case, seed):
    if not (case["graph"] == "er" and case["model"] == "wc" and case["sampler"] == "iis"
            and case["first_step"] == "rejection" and case["kind"] in ("query", "sample")
            and case["samples"] <= 200_000 and case["k"] <= 50):
        return None
    n, T = case["n"], case["samples"]
    src, dst, _ = _edges(case, seed)
    off, csr, tau, w, W, f, prob, alias = _exact_graph(n, src, dst)
    pairs = _exact_sketch(case, off, csr, tau, W, prob, alias)
    js, vs = (pairs // n).cpu().numpy(), (pairs % n).cpu().numpy()
    gap = [(1 << f) - x for x in w.tolist()]

    def influence(cov, sets):
        return (cov * W + T * sum(gap[v] for v in sets)) / (T << f)

    if case["kind"] == "query":
        o, s = _queries(case, seed)
        sets = [s[o[b]:o[b + 1]].tolist() for b in range(case["queries"])]
        cov = [int(np.unique(js[np.isin(vs, x)]).size) for x in sets]
        est = [influence(c, x) for c, x in zip(cov, sets)]
        out = np.array(cov, np.int64), np.array(est, np.float64)
        if case["space"] == "device":
            out = torch.from_numpy(out[0]).cuda(), torch.from_numpy(out[1]).cuda()
        return out
    seeds, cov, est = [], [], []
    covered = np.zeros(T, bool)
    for _ in range(case["k"]):
        delta = np.bincount(vs[~covered[js]], minlength=n).tolist()
        best = max((v for v in range(n) if v not in seeds), key=lambda v: (delta[v] * W + T * gap[v], -v))
        covered[js[vs == best]] = True
        seeds.append(best)
        cov.append(int(covered.sum()))
        est.append(influence(cov[-1], seeds))
    return np.array(seeds, np.int32), np.array(cov, np.int64), np.array(est, np.float64)
