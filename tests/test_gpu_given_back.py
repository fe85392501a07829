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
    assert b["levels"] == 0 and b["lockstep"] == b["given_back"] > 0
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
