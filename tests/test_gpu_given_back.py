"""GPU: batches that the level-mask kernel gives back (too many distance levels for its masks, or a path count
of 2^32) run on the lockstep kernel with what the call has prepared.  Which kernel ran is read from the
context, results are compared with the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_1406_4173_gb300 import gen

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12       # the FP64 bar of the other parity tests


@pytest.fixture(scope="module")
def bc():
    import torch
    import paper_1406_4173_gb300 as m
    from paper_1406_4173_gb300 import _build
    _build.build()
    torch.cuda.set_device(0)
    return m


@pytest.fixture
def ctx(bc):
    c = bc.Context()
    yield c
    c.close()


def rel_err(x, ref):
    x = np.asarray(x.cpu().numpy() if hasattr(x, "cpu") else x, np.float64)
    ref = np.asarray(ref, np.float64)
    return float(np.max(np.abs(x - ref) / np.maximum(np.abs(ref), 1.0))) if x.size else 0.0


def blocks(side, b):
    """Square parts of b x b nodes of a square grid (skeleton weights stay small)."""
    i = np.arange(side * side)
    k = -(-side // b)
    return ((i // side) // b * k + (i % side) // b).astype(np.int32)


def directed_cycle(n, wmax):
    i = np.arange(n, dtype=np.int32)
    w = np.random.default_rng(n).integers(1, wmax + 1, n).astype(np.uint32)
    return gen.EdgeList(n=n, src=i, dst=(i + 1) % n, w=w, directed=True)


# Launches of the attempt: order of the targets apart (the same on both sides), the level-mask pass and its
# sums (with Centrality three per chunk, one chunk here), its combination, and the indicator of the targets.
ATTEMPT = 8


def test_plain_keeps_what_it_prepared(bc, ctx):
    """A deep weighted cycle: as many launches as the FP32 call, which starts on the lockstep kernel, and the attempt."""
    g = directed_cycle(200, 30)
    S = np.arange(0, 200, 3, dtype=np.int32)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    got, st = bc.brandes(G, S, stats=True, ctx=ctx)
    assert rel_err(got, ref) <= FP64_TOL
    b = ctx.last_batches()
    assert b["levels"] == 0 and b["given_back"] == 3 and b["lockstep"] > 0
    _, st32 = bc.brandes(G, S, precision="fp32", stats=True, ctx=ctx)
    assert ctx.last_batches()["given_back"] == 0
    assert st["kernel_launches"] <= st32["kernel_launches"] + ATTEMPT


def test_pp_keeps_its_skeleton(bc, ctx):
    g = gen.with_weights(gen.grid(70, 70), 6, seed=3)   # 269 distance levels, skeleton weights up to 23
    part = blocks(70, 5)
    S = gen.sample_targets(g.n, 80, seed=5)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    got, st = bc.brandes_pp(G, S, part, stats=True, ctx=ctx)
    assert rel_err(got, ref) <= FP64_TOL
    assert ctx.last_batches() == {"levels": 0, "lockstep": 3, "given_back": 3}
    _, st32 = bc.brandes_pp(G, S, part, precision="fp32", stats=True, ctx=ctx)
    assert st["kernel_launches"] <= st32["kernel_launches"] + ATTEMPT


@pytest.mark.parametrize("entry", ["batched", "sssp", "st", "all"])
def test_other_entries(bc, ctx, entry):
    g = gen.path(300)
    part = (np.arange(g.n) // 30).astype(np.int32)   # skeleton weights up to 29
    if entry == "batched":
        gs = [gen.cycle(200), gen.grid(3, 80)]
        arena = bc.build_arena(gs)
        got = bc.brandes_batched(arena, ctx=ctx).cpu().numpy()
        for i, x in enumerate(gs):
            ref, _ = oracle.brandes(x, None)
            assert rel_err(got[arena.node_ptr_host[i]:arena.node_ptr_host[i + 1]], ref) <= FP64_TOL
    elif entry == "sssp":
        src = np.arange(0, g.n, 9, dtype=np.int32)
        d, s = bc.sssp(bc.graph_from_edgelist(g), src, ctx=ctx)
        for i, v in enumerate(src):
            rd, rs, _ = oracle.sssp(g, int(v))
            assert np.array_equal(d[i].cpu().numpy(), rd)
            assert np.array_equal(s[i].cpu().numpy().view(np.uint64), rs)
    else:
        G = bc.graph_from_edgelist(g)
        S = np.arange(0, g.n, 5, dtype=np.int32) if entry == "st" else None
        ref, _ = oracle.brandes(g, S)
        got = bc.brandes_pp_st(G, S, S, part, ctx=ctx) if entry == "st" else bc.brandes_pp_all(G, part, ctx=ctx)
        assert rel_err(got, ref) <= FP64_TOL
    assert ctx.last_batches()["given_back"] > 0


@pytest.mark.parametrize("pp", [False, True])
def test_plan_moves_once(bc, ctx, pp):
    g = gen.with_weights(gen.grid(60, 60), 9, seed=6)   # 322 levels, skeleton weights up to 28
    part = blocks(60, 4)
    S = gen.sample_targets(g.n, 70, seed=5)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    plan = bc.plan_brandes_pp(G, S, part, ctx=ctx) if pp else bc.plan_brandes(G, S, ctx=ctx)
    try:
        for given_back in (3, 0, 0):
            assert rel_err(plan.launch(), ref) <= FP64_TOL
            b = ctx.last_batches()
            assert b["levels"] == 0 and (b["given_back"] > 0) == (given_back > 0)
    finally:
        plan.close()


# ---------------------------------------------------------------------------- levels that are known to be enough
def tree(n, b):
    v = np.arange(1, n, dtype=np.int32)
    return gen.EdgeList(n=n, src=((v - 1) // b).astype(np.int32), dst=v)


def subtrees(n, b, level):
    """Part 0: the top of the tree; then one part per subtree hanging at the level."""
    first = (b ** level - 1) // (b - 1)
    anc = np.arange(n)
    while (anc >= first * b + 1).any():
        anc = np.where(anc >= first * b + 1, (anc - 1) // b, anc)
    return np.where(np.arange(n) < first, 0, anc - first + 1).astype(np.int32)


def star_beside_path(leaves, k):
    i = np.arange(1, leaves + 1)
    p = leaves + 1 + np.arange(k)
    return gen.EdgeList(n=leaves + 1 + k, src=np.concatenate([np.zeros(leaves, np.int64), p[:-1]]).astype(np.int32),
                        dst=np.concatenate([i, p[1:]]).astype(np.int32))


def hub_between_chains(side, com):
    """`side` communities (complete graphs) in a row on either side of a hub of many leaves."""
    src, dst, off = [], [], 0
    for _ in range(2 * side):
        a, b = np.triu_indices(com, 1)
        src.append(a + off), dst.append(b + off)
        if off:
            src.append([off - 1]), dst.append([off])
        off += com
    hub, mid = off, side * com
    src += [[hub, hub], np.full(60, hub)]
    dst += [[mid - 1, mid], hub + 1 + np.arange(60)]
    return gen.EdgeList(n=hub + 61, src=np.concatenate(src).astype(np.int32), dst=np.concatenate(dst).astype(np.int32),
                        part=np.minimum(np.arange(hub + 61) // com, 2 * side).astype(np.int32))


BOUNDED = {
    # levels provided 32, deepest 26, skeleton weights up to 16
    "binary-tree": (tree(16383, 2), subtrees(16383, 2, 4), 100),
    "ternary-tree": (tree(29524, 3), subtrees(29524, 3, 3), 100),
    "hub-between-chains": (hub_between_chains(6, 12), None, 70),
    # levels from the hub: 1; the path beside it: 39, and one more than the 60 that are provided for it at most
    "star-path-40": (star_beside_path(100, 40), np.arange(141) % 3, 100),
    "star-path-60": (star_beside_path(100, 60), np.arange(161) % 3, 100),
}


@pytest.mark.parametrize("name", list(BOUNDED))
def test_bounded_levels_are_enough(bc, ctx, name):
    g, part, k = BOUNDED[name]
    part = (g.part if part is None else part).astype(np.int32)
    S = gen.sample_targets(g.n, k, seed=5)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    for run in (lambda: bc.brandes(G, S, ctx=ctx), lambda: bc.brandes_pp(G, S, part, ctx=ctx)):
        assert rel_err(run(), ref) <= FP64_TOL
        b = ctx.last_batches()
        assert b["levels"] > 0 and b["lockstep"] == 0, b


def test_many_small_components(bc, ctx):
    """Most nodes outside the hub's component: their count says little about the distances."""
    k, m = 300, 12
    src = (np.arange(k)[:, None] * m + np.arange(m - 1)).ravel()
    g = gen.EdgeList(n=k * m + 9, src=np.concatenate([src, np.full(8, k * m)]).astype(np.int32),
                     dst=np.concatenate([src + 1, k * m + 1 + np.arange(8)]).astype(np.int32))
    ref, _ = oracle.brandes(g, None)
    assert rel_err(bc.brandes(bc.graph_from_edgelist(g), None, ctx=ctx), ref) <= FP64_TOL
    assert ctx.last_batches()["lockstep"] == 0


# ---------------------------------------------------------------------------- only the batches that do not fit
def beside(g, h):
    """Disjoint union of two graphs with parts."""
    part = None if g.part is None else np.concatenate([g.part, h.part + g.part.max() + 1]).astype(np.int32)
    return gen.EdgeList(n=g.n + h.n, src=np.concatenate([g.src, h.src + g.n]).astype(np.int32),
                        dst=np.concatenate([g.dst, h.dst + g.n]).astype(np.int32), part=part)


def layers(count, width):
    """Layers of nodes, neighbouring ones completely joined: width^(d - 1) paths at distance d."""
    a, b = (x.ravel() for x in np.meshgrid(np.arange(width), np.arange(width)))
    src = np.concatenate([a + i * width for i in range(count - 1)])
    dst = np.concatenate([b + (i + 1) * width for i in range(count - 1)])
    return gen.EdgeList(n=count * width, src=src.astype(np.int32), dst=dst.astype(np.int32))


# path of 100: four batches, each too deep for the 64 levels of a batched call; 16 layers of eight nodes: 8^11 = 2^33
# paths and more from the first and the last 32 nodes only
@pytest.mark.parametrize("odd,back", [(gen.path(100), 4), (layers(16, 8), 2)], ids=["deep", "counts"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batched_keeps_the_other_graphs(bc, ctx, odd, back, precision):
    gs = [gen.erdos_renyi(n, min(1.0, 6.0 / n), seed=n) for n in (40, 64, 65, 200)] + [odd]
    arena = bc.build_arena(gs)
    got = bc.brandes_batched(arena, precision=precision, ctx=ctx).cpu().numpy()
    for i, g in enumerate(gs):
        ref, _ = oracle.brandes(g, None)
        x = got[arena.node_ptr_host[i]:arena.node_ptr_host[i + 1]]
        assert rel_err(x, ref) <= (FP64_TOL if precision == "fp64" else 2e-6), i
    total = sum(-(-g.n // 32) for g in gs)
    b = ctx.last_batches()
    assert b["levels"] == total - back and b["given_back"] == back and b["lockstep"] >= back


def two_components():
    g = gen.planted_partition(600, 6, 0.06, 0.004, seed=51)
    p = gen.path(300)
    p.part = (np.arange(300) // 30).astype(np.int32)
    return beside(g, p)


@pytest.mark.parametrize("method", ["plain", "plain-fp32", "pp", "pp-chunks", "pp-st", "plan"])
def test_targets_of_a_deep_component(bc, ctx, method):
    g = two_components()
    S = np.concatenate([np.arange(0, 600, 3), np.arange(600, 900, 4)]).astype(np.int32)   # 200 and 75 targets
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    if method.startswith("plain"):
        got = bc.brandes(G, S, precision="fp32" if "32" in method else "fp64", ctx=ctx)
    elif method == "pp-st":
        got = bc.brandes_pp_st(G, S, S, g.part, ctx=ctx)
    elif method == "plan":
        plan = bc.plan_brandes(G, S, ctx=ctx)
        got = plan.launch().cpu().numpy()
        plan.close()
    else:
        got = bc.brandes_pp(G, S, g.part, pp_chunks=int("chunks" in method), ctx=ctx)
    assert rel_err(got, ref) <= (2e-6 if "32" in method else FP64_TOL)
    b = ctx.last_batches()
    if method == "plan":        # moves as a whole
        assert b["levels"] == 0 and b["given_back"] == b["lockstep"] > 0
    else:
        assert 3 <= b["given_back"] <= 3 + (method == "plain-fp32") * 80 and b["lockstep"] >= b["given_back"]
        assert b["levels"] >= 6


def test_paths_from_a_deep_component(bc, ctx):
    g = two_components()
    src = np.concatenate([np.arange(32), 600 + 9 * np.arange(32)]).astype(np.int32)
    d, s = bc.sssp(bc.graph_from_edgelist(g), src, ctx=ctx)
    assert ctx.last_batches() == {"levels": 1, "lockstep": 1, "given_back": 1}
    for i, v in enumerate(src):
        rd, rs, _ = oracle.sssp(g, int(v))
        assert np.array_equal(d[i].cpu().numpy(), rd)
        assert np.array_equal(s[i].cpu().numpy().view(np.uint64), rs)


def test_tables_of_a_deep_part(bc):
    """One part (a path of 300) is too deep for the Dijkstra_SK masks, the others are not."""
    g = two_components()
    part = np.minimum(g.part, 6).astype(np.int32)
    S = np.array([3, 100, 350, 610, 750, 890], np.int32)
    nodes, (u, v, w, mu) = bc.skeleton(bc.graph_from_edgelist(g), S, part)
    rn, (ru, rv, rw, rmu), _ = oracle.skeleton(g, S, part)
    o, ro = np.lexsort((v, u)), np.lexsort((rv, ru))
    assert np.array_equal(np.sort(nodes), np.sort(rn))
    for x, rx in ((u, ru), (v, rv), (w, rw), (mu, rmu)):
        assert np.array_equal(np.asarray(x)[o].astype(np.uint64), np.asarray(rx)[ro].astype(np.uint64))


# ---------------------------------------------------------------------------- levels without an order of the targets
def community_chain(count, size):
    g = [gen.erdos_renyi(size, 8.0 / size, seed=60 + i) for i in range(count)]
    src = [x.src + i * size for i, x in enumerate(g)] + [np.arange(1, count) * size]
    dst = [x.dst + i * size for i, x in enumerate(g)] + [np.arange(1, count) * size - 1]
    lo, hi = (f(np.concatenate(src), np.concatenate(dst)).astype(np.int32) for f in (np.minimum, np.maximum))
    return gen.EdgeList(n=count * size, src=lo, dst=hi)


def test_few_unordered_targets_of_a_long_graph(bc, ctx):
    """More than 64 levels, nothing known about them, few batches: the masks hold them all."""
    g = community_chain(20, 60)
    G = bc.graph_from_edgelist(g)
    for S, kw in ((gen.sample_targets(g.n, 60, seed=5), {}), (gen.sample_targets(g.n, 200, seed=5), {"order_sources": False})):
        ref, _ = oracle.brandes(g, S)
        assert max(x for x in oracle.sssp(g, int(S[0]))[0] if x < 2**31 - 1) > 64
        assert rel_err(bc.brandes(G, S, ctx=ctx, **kw), ref) <= FP64_TOL
        assert ctx.last_batches()["lockstep"] == 0


@pytest.mark.parametrize("count,size,route", [(30, 310, "lockstep"), (8, 1100, "levels")])
def test_many_unordered_targets(bc, ctx, count, size, route):
    """Large calls in the given order: the levels from the hub decide as they do for ordered calls."""
    g = community_chain(count, size)
    S = None
    ref, _ = oracle.brandes(g, S)
    got = bc.brandes(bc.graph_from_edgelist(g), S, order_sources=False, ctx=ctx)
    assert rel_err(got, ref) <= FP64_TOL
    b = ctx.last_batches()
    assert b["given_back"] == 0 and b[route] > 0 and sum(b.values()) == b[route]


@pytest.mark.parametrize("hubs,leaves", [(8, 150), (40, 40), (70, 33)])
@pytest.mark.parametrize("k", [40, 64, 400])
def test_hubs_in_single_tiles(bc, ctx, hubs, leaves, k):
    """A row of hubs with neighbouring ids: tiles of thousands of arcs among tiles of 32, taken in parts."""
    n = hubs * (leaves + 1)
    leaf = np.arange(hubs, n)
    g = gen.EdgeList(n=n, src=np.concatenate([np.arange(hubs - 1), (leaf - hubs) % hubs]).astype(np.int32),
                     dst=np.concatenate([np.arange(1, hubs), leaf]).astype(np.int32))
    S = gen.sample_targets(n, k, seed=6)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    assert rel_err(bc.brandes(G, S, ctx=ctx), ref) <= FP64_TOL
    assert rel_err(bc.brandes(G, S, precision="fp32", ctx=ctx), ref) <= 2e-6
    d, s = bc.sssp(G, S[:33], ctx=ctx)
    for i, v in enumerate(S[:33]):
        rd, rs, _ = oracle.sssp(g, int(v))
        assert np.array_equal(d[i].cpu().numpy(), rd)
        assert np.array_equal(s[i].cpu().numpy().view(np.uint64), rs)


# ---------------------------------------------------------------------------- plans of a rewritten graph
def spine(length, n):
    """A path of `length` nodes and n - length leaves, spread over it: n - 1 edges."""
    leaf = np.arange(length, n)
    src = np.concatenate([np.arange(length - 1), leaf % length])
    dst = np.concatenate([np.arange(1, length), leaf])
    return gen.EdgeList(n=n, src=src.astype(np.int32), dst=dst.astype(np.int32))


def rewrite(bc, G, g):
    new = bc.graph_from_edgelist(g)
    G.row_ptr.copy_(new.row_ptr)
    G.col.copy_(new.col)


@pytest.mark.parametrize("order_sources", [True, False])
def test_plan_follows_a_deeper_graph_and_back(bc, ctx, order_sources):
    flat, deep, deeper = gen.star(500), spine(60, 500), spine(110, 500)
    S = gen.sample_targets(500, 90, seed=2)
    G = bc.graph_from_edgelist(flat)
    plan = bc.plan_brandes(G, S, order_sources=order_sources, ctx=ctx)
    try:
        for g in (flat, deep, deep, flat, deeper, flat, deep):
            rewrite(bc, G, g)
            assert rel_err(plan.launch(), oracle.brandes(g, S)[0]) <= FP64_TOL
            b = ctx.last_batches()
            assert b["lockstep"] == 0 and b["given_back"] == 0, b
        # past what the masks can hold: moves to the lockstep kernel, and is right on it
        for g in (gen.path(500), flat):
            rewrite(bc, G, g)
            assert rel_err(plan.launch(), oracle.brandes(g, S)[0]) <= FP64_TOL
            assert ctx.last_batches()["levels"] == 0
    finally:
        plan.close()


@pytest.mark.parametrize("tail", [20, 300])
@pytest.mark.parametrize("sources", [1, 33])
def test_early_test_for_deep_graphs(bc, ctx, tail, sources):
    """The tests an eighth and a quarter of the way: a grid past the levels is given up, a graph with a tail within them
    is not, also from a single source; Dijkstra_SK tables of a deep part, too."""
    deep = gen.with_weights(gen.grid(60, 60), 16, seed=71)
    e = gen.erdos_renyi(700, 0.01, seed=72)
    t = np.concatenate([[0], e.n + np.arange(tail)]).astype(np.int32)
    within = gen.with_weights(gen.EdgeList(n=e.n + tail, src=np.concatenate([e.src, t[:-1]]),
                                           dst=np.concatenate([e.dst, t[1:]])), 9 if tail < 100 else 1, seed=73)
    for g, served in ((deep, False), (within, tail < 100)):
        src = np.arange(0, g.n, g.n // sources, dtype=np.int32)[:sources]
        d, s = bc.sssp(bc.graph_from_edgelist(g), src, ctx=ctx)
        assert (ctx.last_batches()["levels"] > 0) == served
        for i, v in enumerate(src):
            rd, rs, _ = oracle.sssp(g, int(v))
            assert np.array_equal(d[i].cpu().numpy(), rd)
            assert np.array_equal(s[i].cpu().numpy().view(np.uint64), rs)
    part = (np.arange(deep.n) // 1200).astype(np.int32)
    S = gen.sample_targets(deep.n, 6, seed=5)
    ref, _ = oracle.brandes(deep, S)
    assert rel_err(bc.brandes_pp(bc.graph_from_edgelist(deep), S, part, ctx=ctx), ref) <= FP64_TOL


@pytest.mark.parametrize("method", ["plain", "pp"])
def test_few_batches_go_together(bc, ctx, method):
    """Three of six batches do not fit: the lockstep kernel takes all six at once."""
    g = two_components()
    S = np.concatenate([np.arange(0, 600, 6), np.arange(600, 900, 4)]).astype(np.int32)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    got = bc.brandes(G, S, ctx=ctx) if method == "plain" else bc.brandes_pp(G, S, g.part, ctx=ctx)
    assert rel_err(got, ref) <= FP64_TOL
    b = ctx.last_batches()
    assert b["levels"] == 0 and b["given_back"] == 6


def test_long_row_of_a_weighted_graph(bc, ctx):
    g = gen.with_weights(gen.star(9000), 20, seed=9)
    S = gen.sample_targets(g.n, 70, seed=9)
    ref, _ = oracle.brandes(g, S)
    assert rel_err(bc.brandes(bc.graph_from_edgelist(g), S, ctx=ctx), ref) <= FP64_TOL
    b = ctx.last_batches()
    assert b["levels"] == 0 and b["given_back"] == 0


def test_unreachable_pairs_are_not_depth(bc, ctx):
    """A directed graph without cycles: most pairs are never reached, which the test for deep graphs must not take for
    levels still to come."""
    r = np.random.default_rng(2)
    n = 8000
    u = r.integers(0, n, 5 * n)
    v = (u + r.integers(1, n, 5 * n)) % n
    key = np.unique(np.minimum(u, v).astype(np.int64) * n + np.maximum(u, v))
    g = gen.EdgeList(n=n, src=(key // n).astype(np.int32), dst=(key % n).astype(np.int32),
                     w=r.integers(1, 10, len(key)).astype(np.uint32), directed=True)
    S = gen.sample_targets(n, 100, seed=4)
    ref, _ = oracle.brandes(g, S)
    assert rel_err(bc.brandes(bc.graph_from_edgelist(g), S, ctx=ctx), ref) <= FP64_TOL
    assert ctx.last_batches()["levels"] > 0
