"""The calls whose speed matters to a user of this library, as timed cases.

Each case is one pass through a public entry point on inputs of the families that the library's
benchmark and tests use: Chung-Lu graphs with planted communities, planted partitions, directed
graphs with integer weights, batches of small random graphs.  Graphs are drawn on the GPU from
the seed; a user's program holds the CSR graph, the target set and the partition before it asks
for betweenness, so these are prepared; the edge list is what a user holds before csr_build.
"""
import math

import numpy as np
import torch

import paper_1406_4173_gb300 as bc
from paper_1406_4173_gb300 import api


def listed():
    """Sizes: S = 0 means every node is a target."""
    return [
        # a small network, every node a target: launches and latency decide
        dict(name="plain_planted_2k", kind="plain", family="planted", n=2000, deg=6.0, com=250, intra=0.85, wmax=0,
             directed=False, S=0, precision="fp64"),
        # the ordinary case: full betweenness of a network with communities and hubs
        dict(name="plain_chunglu_50k", kind="plain", family="chunglu", n=50000, deg=10.0, com=1000, intra=0.9, wmax=0,
             directed=False, S=0, precision="fp64"),
        # the largest graph of the benchmark, 4,096 targets
        dict(name="plain_chunglu_1m", kind="plain", family="chunglu", n=1000000, deg=16.0, com=1000, intra=0.85,
             wmax=0, directed=False, S=4096, precision="fp64"),
        # the faster, less exact mode, on an odd size
        dict(name="plain_fp32_20011", kind="plain", family="chunglu", n=20011, deg=12.0, com=700, intra=0.9, wmax=0,
             directed=False, S=0, precision="fp32"),
        # road- or latency-like weights on a directed network
        dict(name="plain_directed_w16", kind="plain", family="chunglu", n=100000, deg=12.0, com=500, intra=0.9,
             wmax=16, directed=True, S=2000, precision="fp64"),
        # Brandes++ on a network whose communities have many frontiers: the whole pipeline, middle size
        dict(name="pp_chunglu_100k", kind="pp", family="chunglu", n=100000, deg=16.0, com=1000, intra=0.85, wmax=0,
             directed=False, S=512, precision="fp64"),
        # the same at the benchmark's largest graph
        dict(name="pp_chunglu_1m", kind="pp", family="chunglu", n=1000000, deg=16.0, com=1000, intra=0.85, wmax=0,
             directed=False, S=2048, precision="fp64"),
        # Brandes++ where the partition cuts few edges (the paper's regime) and targets are few
        dict(name="pp_planted_200k", kind="pp", family="planted", n=200000, deg=10.0, com=2000, intra=0.998, wmax=0,
             directed=False, S=200, precision="fp64"),
        # thousands of independent graphs in one call
        dict(name="batched_er_4096", kind="batched", graphs=4096, median=512, deg=8.0, precision="fp64"),
        # distances and path counts from a few sources of a weighted directed network
        dict(name="sssp_directed_w16", kind="sssp", family="chunglu", n=20000, deg=12.0, com=500, intra=0.9, wmax=16,
             directed=True, S=64),
        # a captured evaluation, replayed (a service that asks for the same graph again)
        dict(name="plan_chunglu_10k", kind="plan", family="chunglu", n=10000, deg=10.0, com=1000, intra=0.9, wmax=0,
             directed=False, S=0, precision="fp64"),
        # what comes before everything else: the graph from its edge list
        dict(name="csr_build_8m", kind="csr", family="chunglu", n=1000000, deg=16.0, com=1000, intra=0.85, wmax=0,
             directed=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["plain", "plain", "plain", "pp", "pp", "batched", "sssp", "plan", "csr"])
    if kind == "batched":
        return dict(kind=kind, graphs=int(_log(rng, 16, 3000)), median=int(_log(rng, 64, 600)),
                    deg=round(rng.uniform(3, 12), 1), precision=rng.choice(["fp64", "fp64", "fp32"]))
    weighted = kind in ("plain", "pp", "sssp") and rng.random() < 0.3
    top = {"plain": 600000, "pp": 300000, "sssp": 100000, "plan": 50000, "csr": 1000000}[kind]
    n = int(_log(rng, 600, top if not weighted else min(top, 60000)))
    deg = round(rng.uniform(5, 18), 1)
    family = rng.choice(["chunglu", "chunglu", "planted"])
    case = dict(kind=kind, family=family, n=n, deg=deg, com=int(min(n // 4, _log(rng, 100, 2000))),
                intra=rng.choice([0.8, 0.85, 0.9, 0.95]), wmax=rng.choice([7, 9, 16]) if weighted else 0,
                directed=weighted and rng.random() < 0.5 or (kind == "plain" and rng.random() < 0.2))
    if kind == "csr":
        return case
    # sources x arcs, bounded so that no draw costs more than the largest listed case
    arcs = n * deg
    most = {"plain": 3e9 if weighted else 2.5e10, "pp": 5e8 if weighted else 2e9, "sssp": 2e8, "plan": 2e9}[kind]
    S = int(_log(rng, 16, max(17, min(n, most / arcs, 300 if kind == "sssp" else n))))
    case["S"] = 0 if kind in ("plain", "plan") and n * arcs <= most and rng.random() < 0.5 else S
    if kind != "sssp":
        case["precision"] = "fp32" if rng.random() < 0.15 else "fp64"
    return case


# ----------------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _unique_in_order(keys, count):
    """The first `count` distinct keys in the order drawn."""
    k, order = torch.sort(keys, stable=True)
    first = torch.ones_like(k, dtype=torch.bool)
    first[1:] = k[1:] != k[:-1]
    at = torch.sort(order[first]).values[:count]
    return keys[at]


def _edges(c, seed):
    """(src, dst, weights or None, community of each node), int32 on the GPU; undirected: each edge once."""
    g = _generator(seed)
    n, com = c["n"], max(2, c["com"])
    dev = "cuda"
    part = torch.arange(n, device=dev) // com
    lo, hi = part * com, torch.clamp((part + 1) * com, max=n)
    m = int(n * c["deg"] * (1.0 if c["directed"] else 0.5))
    if c["family"] == "chunglu":
        # expected degrees: power law (exponent 2.3), scaled to the mean degree, capped at sqrt(mean n)
        x = (1.0 - torch.rand(n, device=dev, dtype=torch.float64, generator=g)) ** (-1.0 / 1.3)
        x = torch.clamp(x * (c["deg"] / x.mean()), max=math.sqrt(c["deg"] * n))
        cum = torch.cat([torch.zeros(1, device=dev, dtype=torch.float64), torch.cumsum(x, 0)])
    else:
        cum = torch.arange(n + 1, device=dev, dtype=torch.float64)

    def pick(a, b):
        r = torch.rand(a.numel(), device=dev, dtype=torch.float64, generator=g)
        t = cum[a] + r * (cum[b] - cum[a])
        return torch.minimum(torch.maximum(torch.searchsorted(cum, t, right=True) - 1, a), b - 1)

    got = torch.zeros(0, dtype=torch.int64, device=dev)
    for _ in range(12):
        need = m - got.numel()
        if need <= 0:
            break
        k = int(need * 1.2) + 64
        u = pick(torch.zeros(k, dtype=torch.int64, device=dev), torch.full((k,), n, device=dev))
        inside = torch.rand(k, device=dev, generator=g) < c["intra"]
        v = pick(torch.where(inside, lo[u], 0), torch.where(inside, hi[u], n))
        ok = (u != v) & (inside | (part[u] != part[v]))
        u, v = u[ok], v[ok]
        if not c["directed"]:
            u, v = torch.minimum(u, v), torch.maximum(u, v)
        got = _unique_in_order(torch.cat([got, u * n + v]), m)
    src, dst = (got // n).int(), (got % n).int()
    w = None
    if c["wmax"]:
        w = torch.randint(1, c["wmax"] + 1, (got.numel(),), device=dev, dtype=torch.int32, generator=g)
    return src, dst, w, part.int()


def _targets(c, seed):
    if not c["S"] or c["S"] >= c["n"]:
        return None
    g = _generator(seed + 5)
    return torch.sort(torch.randperm(c["n"], device="cuda", generator=g)[: c["S"]]).values.int()


def _arena(c, seed):
    """Node offsets and edges of the batch: sizes log-normal (sigma 0.75) in [64, 4096] (the same ones for every
    seed, so that outputs keep their shape), mean degree c["deg"]."""
    sizes = np.random.default_rng(c["graphs"]).normal(math.log(c["median"]), 0.75, c["graphs"])
    ns = np.clip(np.round(np.exp(sizes)), 64, 4096).astype(np.int64)
    ptr = np.concatenate([[0], np.cumsum(ns)]).astype(np.int64)
    g = _generator(seed)
    ms = np.round(ns * c["deg"] / 2).astype(np.int64)
    nn = torch.repeat_interleave(torch.as_tensor(ns, device="cuda"), torch.as_tensor(ms, device="cuda"))
    off = torch.repeat_interleave(torch.as_tensor(ptr[:-1], device="cuda"), torch.as_tensor(ms, device="cuda"))
    u = (torch.rand(nn.numel(), device="cuda", dtype=torch.float64, generator=g) * nn).long()
    v = (torch.rand(nn.numel(), device="cuda", dtype=torch.float64, generator=g) * nn).long()
    ok = u != v
    a, b = (torch.minimum(u, v) + off)[ok], (torch.maximum(u, v) + off)[ok]
    keys = torch.unique(a * int(ptr[-1]) + b)
    return ptr, (keys // int(ptr[-1])).int(), (keys % int(ptr[-1])).int()


def prepare(case, seed):
    c = case
    if c["kind"] == "batched":
        ptr, src, dst = _arena(c, seed)
        G = bc.csr_build(int(ptr[-1]), src, dst, None, False)
        return dict(kind=c["kind"], arena=api.Arena(torch.as_tensor(ptr, device="cuda"), ptr, G),
                    precision=c["precision"])
    src, dst, w, part = _edges(c, seed)
    st = dict(kind=c["kind"])
    if c["kind"] == "csr":
        st.update(n=c["n"], src=src, dst=dst, w=w, directed=c["directed"])
        return st
    G = bc.csr_build(c["n"], src, dst, w, c["directed"])
    S = _targets(c, seed)
    st.update(G=G, S=S, precision=c.get("precision"))
    if c["kind"] == "pp":
        st.update(part=part, k=-(-c["n"] // max(2, c["com"])))
    if c["kind"] == "sssp":
        st["S"] = S if S is not None else torch.arange(c["n"], dtype=torch.int32, device="cuda")
    if c["kind"] == "plan":
        st["plan"] = bc.plan_brandes(G, S, precision=c["precision"])
    return st


def run(state):
    s = state
    if s["kind"] == "plain":
        return bc.brandes(s["G"], s["S"], precision=s["precision"])
    if s["kind"] == "pp":
        return bc.brandes_pp(s["G"], s["S"], s["part"], s["k"], precision=s["precision"])
    if s["kind"] == "batched":
        return bc.brandes_batched(s["arena"], precision=s["precision"])
    if s["kind"] == "sssp":
        return bc.sssp(s["G"], s["S"])
    if s["kind"] == "plan":
        return s["plan"].launch()
    G = bc.csr_build(s["n"], s["src"], s["dst"], s["w"], s["directed"])
    return [G.row_ptr, G.col] + ([] if G.w is None else [G.w])


def work(case):
    c = case
    if c["kind"] == "batched":
        nodes = c["graphs"] * c["median"] * 1.32
        # mean of n^2 over mean of n of the log-normal: sources per node
        pairs = c["graphs"] * (c["median"] ** 2) * 3.0 * c["deg"]
        return dict(bytes=nodes * (8 + 8) + nodes * c["deg"] * 4, flops=3 * pairs)
    arcs = c["n"] * c["deg"]
    graph = 8 * (c["n"] + 1) + arcs * (8 if c["wmax"] else 4)
    if c["kind"] == "csr":
        edges = arcs * (1.0 if c["directed"] else 0.5)
        return dict(bytes=graph + edges * (12 if c["wmax"] else 8), flops=0)
    S = c["S"] or c["n"]
    if c["kind"] == "sssp":
        return dict(bytes=graph + 12.0 * S * c["n"], flops=2.0 * S * arcs)
    # each source tests each arc once, and adds a count and a dependency over about half of them each
    return dict(bytes=graph + 4 * S + 8 * c["n"], flops=3.0 * S * arcs)


# ----------------------------------------------------------------------------- in 64 bits, by sparse products
def _csr(rows, cols, n):
    key = torch.sort(rows.long() * n + cols.long()).values
    r, col = key // n, key % n
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    one = torch.ones(col.numel(), dtype=torch.float64, device="cuda")
    return torch.sparse_csr_tensor(rp, col, one, size=(n, n))


def _dependencies(n, u, v, w, wmax, first, is_target):
    """Sum over the columns j of the dependencies of the source first[j] (-1: none) on every node; arcs u -> v."""
    nw = wmax or 1
    into = [_csr(v if w is None else v[w == k], u if w is None else u[w == k], n) for k in range(1, nw + 1)]
    out = [_csr(u if w is None else u[w == k], v if w is None else v[w == k], n) for k in range(1, nw + 1)]
    b = first.shape[1]
    seen = torch.full((n, b), -1, dtype=torch.int16, device="cuda")
    start = torch.zeros((n, b), dtype=torch.float64, device="cuda")
    rows, cols = torch.nonzero(first, as_tuple=True)
    start[rows, cols] = 1.0
    seen[rows, cols] = 0
    sig = start.clone()
    ring, last, d = [start], 0, 0
    while d - last < nw:
        d += 1
        x = None
        for k in range(1, min(nw, len(ring)) + 1):
            if ring[-k] is not None:
                y = into[k - 1] @ ring[-k]
                x = y if x is None else x.add_(y)
        new = None
        if x is not None:
            hit = (seen < 0) & (x > 0)
            if bool(hit.any()):
                seen[hit] = d
                new = torch.where(hit, x, 0.0)
                sig += new
                last = d
        ring = (ring + [new])[-nw:]
    delta = torch.zeros_like(sig)
    target = is_target.double()[:, None]
    back = []
    for d in range(last, -1, -1):
        at = seen == d
        for k in range(1, min(nw, len(back)) + 1):
            y = out[k - 1] @ back[-k]
            delta = torch.where(at, torch.addcmul(delta, sig, y), delta)
        back = (back + [torch.where(at, (target + delta) / torch.clamp(sig, min=1.0), 0.0)])[-nw:]
    return torch.where(seen > 0, delta, 0.0).sum(1)


def exact(case, seed):
    c = case
    if c["kind"] in ("sssp", "csr"):
        return None   # whole numbers
    if c["kind"] == "batched":
        ptr, src, dst = _arena(c, seed)
        n = int(ptr[-1])
        if n * 8.0 * np.diff(ptr).max() > 1.2e11:
            return None
        u, v = torch.cat([src, dst]), torch.cat([dst, src])
        local = torch.arange(n, device="cuda") - torch.repeat_interleave(
            torch.as_tensor(ptr[:-1], device="cuda"), torch.as_tensor(np.diff(ptr), device="cuda"))
        size = torch.repeat_interleave(torch.as_tensor(np.diff(ptr), device="cuda"),
                                       torch.as_tensor(np.diff(ptr), device="cuda"))
        total = torch.zeros(n, dtype=torch.float64, device="cuda")
        top, j0 = int(np.diff(ptr).max()), 0
        while j0 < top:
            # the graphs that have a node j0, as a graph of their own
            keep = size > j0
            kept = int(keep.sum())
            b = int(max(1, min(top - j0, 2e8 // kept)))
            ids = torch.cumsum(keep.long(), 0) - 1
            e = keep[u.long()]
            cols = torch.arange(j0, j0 + b, device="cuda")
            total[keep] += _dependencies(kept, ids[u[e].long()], ids[v[e].long()], None, 0,
                                         local[keep][:, None] == cols[None, :],
                                         torch.ones(kept, dtype=torch.bool, device="cuda"))
            j0 += b
        return total / 2
    src, dst, w, _ = _edges(c, seed)
    n = c["n"]
    S = _targets(c, seed)
    S = torch.arange(n, device="cuda") if S is None else S.long()
    if S.numel() * n * c["deg"] * max(1, c["wmax"]) ** 0.7 > 4e10:
        return None   # too slow this way
    if c["directed"]:
        u, v = src, dst
    else:
        u, v = torch.cat([src, dst]), torch.cat([dst, src])
        w = None if w is None else torch.cat([w, w])
    is_target = torch.zeros(n, dtype=torch.bool, device="cuda")
    is_target[S] = True
    total = torch.zeros(n, dtype=torch.float64, device="cuda")
    b = int(max(16, min(1024, 1e8 // n)))
    for j in range(0, S.numel(), b):
        s = S[j:j + b]
        first = torch.zeros((n, s.numel()), dtype=torch.bool, device="cuda")
        first[s, torch.arange(s.numel(), device="cuda")] = True
        total += _dependencies(n, u, v, w, c["wmax"], first, is_target)
    return total if c["directed"] else total / 2
