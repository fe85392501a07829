"""GPU parity of the level-mask kernel (plain Brandes and batched graphs in FP64) at the sizes where
its tiling can go wrong, against the CPU oracle: node counts around a tile of 32 rows, source counts
around a batch of 32, degrees around the 256-arc round of a tile, unreachable nodes, depths and path
counts past what it serves (the call then reruns on the lockstep kernel), weights around its limit.
"""
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


def rel_err(x, ref):
    x = np.asarray(x, np.float64)
    ref = np.asarray(ref, np.float64)
    return float(np.max(np.abs(x - ref) / np.maximum(np.abs(ref), 1.0))) if x.size else 0.0


def union(*graphs):
    """Disjoint union of edge lists (unreachable pairs)."""
    off, src, dst = 0, [], []
    for g in graphs:
        src.append(g.src + off)
        dst.append(g.dst + off)
        off += g.n
    return gen.EdgeList(n=off, src=np.concatenate(src).astype(np.int32), dst=np.concatenate(dst).astype(np.int32))


def wheel_of(deg, extra, seed):
    """One hub of the given degree over a sparse random graph of its neighbours."""
    g = gen.erdos_renyi(deg, min(1.0, extra / deg), seed=seed)
    src = np.concatenate([np.zeros(deg, np.int32), g.src + 1]).astype(np.int32)
    dst = np.concatenate([np.arange(1, deg + 1, dtype=np.int32), g.dst + 1]).astype(np.int32)
    return gen.EdgeList(n=deg + 1, src=src, dst=dst)


CASES = {
    **{f"n{n}": (gen.erdos_renyi(n, min(1.0, 3.5 / n), seed=n), None) for n in (2, 3, 31, 32, 33, 63, 64, 65, 97)},
    **{f"S{k}": (gen.planted_partition(300, 5, 0.06, 0.004, seed=4), k) for k in (2, 31, 32, 33, 64, 65)},
    **{f"deg{d}": (wheel_of(d, 2.0, seed=d), None) for d in (255, 256, 257, 300, 513)},
    "star": (gen.star(700), None),
    "complete": (gen.complete(90), None),
    "islands": (union(gen.path(40), gen.complete(9), gen.star(33), gen.cycle(50)), None),
    "path-deep": (gen.path(400), None),
    "grid-counts": (gen.grid(34, 34), 70),
    "w-limit": (gen.planted_partition(400, 4, 0.03, 0.004, seed=5, wmax=32), None),
    "w-past-limit": (gen.planted_partition(400, 4, 0.03, 0.004, seed=6, wmax=33), None),
    "w-deep": (gen.with_weights(gen.grid(20, 20), 32, seed=7), None),
    "directed-w": (gen.chung_lu_communities(500, [125] * 4, 2.3, 5.0, 0.85, seed=8, directed=True, wmax=9), None),
    "directed": (gen.chung_lu_communities(500, [125] * 4, 2.3, 5.0, 0.85, seed=9, directed=True), 77),
}


@pytest.mark.parametrize("name", list(CASES))
def test_levels_match_oracle(bc, name):
    g, k = CASES[name]
    S = None if k is None else gen.sample_targets(g.n, k, seed=3)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    assert rel_err(bc.brandes(G, S).cpu().numpy(), ref) <= FP64_TOL
    # the same batches in another order of the sources, and as two shards
    assert rel_err(bc.brandes(G, S, order_sources=False).cpu().numpy(), ref) <= FP64_TOL
    parts = [bc.brandes(G, S, shard=(r, 2)).cpu().numpy() for r in range(2)]
    assert rel_err(parts[0] + parts[1], ref) <= FP64_TOL


def test_levels_batched(bc):
    gs = [gen.erdos_renyi(n, min(1.0, 4.0 / n), seed=n) for n in (1, 2, 31, 32, 33, 64, 65, 130, 257)]
    gs += [gen.path(300), gen.star(290)]
    arena = bc.build_arena(gs)
    got = bc.brandes_batched(arena).cpu().numpy()
    for i, g in enumerate(gs):
        ref, _ = oracle.brandes(g, None)
        x = got[arena.node_ptr_host[i]:arena.node_ptr_host[i + 1]]
        assert rel_err(x, ref) <= FP64_TOL, i


# Brandes_SK on the level-mask kernel: 64-bit counts, multiplicities, distance rows for the Centrality
# step; skeleton rows below and above the 256-arc round, batches of 1 to 65 sources, chunks of batches
PP_CASES = {
    "planted": (gen.planted_partition(600, 6, 0.05, 0.004, seed=21), 65),
    "planted-w": (gen.planted_partition(500, 5, 0.05, 0.004, seed=22, wmax=9), 33),
    "dense-cliques": (gen.planted_partition(800, 2, 0.02, 0.006, seed=23), 32),
    "directed-w": (gen.chung_lu_communities(500, [125] * 4, 2.3, 6.0, 0.85, seed=24, directed=True, wmax=7), 64),
    "w-past-limit": (gen.planted_partition(400, 4, 0.05, 0.004, seed=25, wmax=40), 40),
    "all-targets": (gen.planted_partition(300, 5, 0.06, 0.004, seed=26), None),
}


@pytest.mark.parametrize("name", list(PP_CASES))
def test_levels_skeleton_matches_oracle(bc, name):
    g, k = PP_CASES[name]
    S = None if k is None else gen.sample_targets(g.n, k, seed=3)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    for kw in ({}, {"pp_chunks": 1}, {"order_sources": False}):
        got = bc.brandes_pp(G, S, g.part, **kw).cpu().numpy()
        assert rel_err(got, ref) <= FP64_TOL, kw


@pytest.mark.parametrize("name", ["n33", "n65", "S33", "star", "islands", "path-deep", "grid-counts", "w-limit",
                                  "w-past-limit", "w-deep", "directed-w", "directed"])
def test_levels_paths_match_oracle(bc, name):
    """Distances and counts, bit for bit; 33 sources, one of them twice."""
    g, _ = CASES[name]
    src = np.concatenate([np.arange(0, g.n, max(1, g.n // 32))[:32], [0]]).astype(np.int32)
    d, s = bc.sssp(bc.graph_from_edgelist(g), src)
    d, s = d.cpu().numpy(), s.cpu().numpy().view(np.uint64)
    for i, v in enumerate(src):
        rd, rs, _ = oracle.sssp(g, int(v))
        assert np.array_equal(d[i], rd), i
        assert np.array_equal(s[i], rs), i


TABLE_CASES = {
    "planted": (gen.planted_partition(400, 4, 0.05, 0.006, seed=31), 20),
    "planted-w": (gen.planted_partition(400, 4, 0.05, 0.006, seed=32, wmax=9), 33),
    "one-big-part": (gen.planted_partition(700, 2, 0.03, 0.004, seed=33), 10),
    "directed-w": (gen.chung_lu_communities(300, [75] * 4, 2.3, 6.0, 0.85, seed=34, directed=True, wmax=7), 15),
    "deep-part": (gen.path(300), 5),          # a part deeper than the kernel serves: the lockstep tables
}


@pytest.mark.parametrize("name", list(TABLE_CASES))
def test_tables_give_the_oracle_skeleton(bc, name):
    """Dijkstra_SK on the level-mask kernel (frontier parents excluded from the counts): the skeleton's arcs,
    weights and multiplicities, exactly."""
    g, k = TABLE_CASES[name]
    part = g.part if g.part is not None else (np.arange(g.n) * 2 // g.n).astype(np.int32)
    S = gen.sample_targets(g.n, k, seed=4)
    nodes, (u, v, w, mu) = bc.skeleton(bc.graph_from_edgelist(g), S, part)
    rn, (ru, rv, rw, rmu), _ = oracle.skeleton(g, S, part)
    o, ro = np.lexsort((v, u)), np.lexsort((rv, ru))
    assert np.array_equal(np.sort(nodes), np.sort(rn))
    for x, rx in ((u, ru), (v, rv), (w, rw), (mu, rmu)):
        assert np.array_equal(np.asarray(x)[o].astype(np.uint64), np.asarray(rx)[ro].astype(np.uint64))


def spoked(k, wmax=None):
    """Part 0: a hub and its k neighbours, each tied to one node of a ring (part 1): the hub is a
    non-frontier node with k frontiers that all reach it directly."""
    i = np.arange(1, k + 1)
    src = np.concatenate([np.zeros(k, np.int64), i, i + k])
    dst = np.concatenate([i, i + k, np.roll(i + k, -1)])
    lo, hi = np.minimum(src, dst), np.maximum(src, dst)
    g = gen.EdgeList(n=2 * k + 1, src=lo.astype(np.int32), dst=hi.astype(np.int32),
                     part=(np.arange(2 * k + 1) > k).astype(np.int32))
    return g if wmax is None else gen.with_weights(g, wmax, seed=k)


@pytest.mark.parametrize("k", [3, 31, 32, 33, 127, 128, 129, 300])
@pytest.mark.parametrize("wmax", [None, 5])
def test_centrality_list_lengths(bc, k, wmax):
    """Centrality's frontier lists around its chunk of 32 and its stage of 128 entries."""
    g = spoked(k, wmax)
    S = np.arange(k + 1, 2 * k + 1, max(1, k // 40), dtype=np.int32)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    got = bc.brandes_pp(G, S, g.part).cpu().numpy()
    assert rel_err(got, ref) <= FP64_TOL
    f32 = bc.brandes_pp(G, S, g.part, precision="fp32").cpu().numpy()
    assert rel_err(f32, ref) <= 2e-6   # the FP32 bar of the other parity tests on small graphs


@pytest.mark.parametrize("deg", [257, 383, 384, 385, 512, 1025])
@pytest.mark.parametrize("wmax", [None, 9])
def test_long_rows(bc, deg, wmax):
    """Rows of more than 256 arcs around the 128 arcs that are looked at together."""
    g = wheel_of(deg, 2.0, seed=deg)
    g = g if wmax is None else gen.with_weights(g, wmax, seed=deg)
    S = gen.sample_targets(g.n, 40, seed=3)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    assert rel_err(bc.brandes(G, S).cpu().numpy(), ref) <= FP64_TOL
    f32 = bc.brandes(G, S, precision="fp32").cpu().numpy()
    assert rel_err(f32, ref) <= 2e-6   # the FP32 bar of the other parity tests on small graphs
    d, s = bc.sssp(G, S[:3])
    for i, v in enumerate(S[:3]):
        rd, rs, _ = oracle.sssp(g, int(v))
        assert np.array_equal(d[i].cpu().numpy(), rd)
        assert np.array_equal(s[i].cpu().numpy().view(np.uint64), rs)


@pytest.mark.parametrize("k", [1, 227, 228, 255, 256, 257])
def test_source_order_small_levels(bc, k):
    """Levels around the 256 nodes and 2,048 arcs that one block takes alone: a hub, k children with eight
    leaves each, and a chain (every node a target, so a node missing from the order shows)."""
    i = np.arange(1, k + 1)
    leaves = k + 1 + np.arange(8 * k)
    tail = np.concatenate([[0], 9 * k + 1 + np.arange(40)])
    src = np.concatenate([np.zeros(k, np.int64), np.repeat(i, 8), tail[:-1]])
    dst = np.concatenate([i, leaves, tail[1:]])
    g = gen.EdgeList(n=9 * k + 41, src=src.astype(np.int32), dst=dst.astype(np.int32))
    ref, _ = oracle.brandes(g, None)
    assert rel_err(bc.brandes(bc.graph_from_edgelist(g), None).cpu().numpy(), ref) <= FP64_TOL


def with_tail(g, k):
    """g and a path of k more nodes from its node 0."""
    t = np.concatenate([[0], g.n + np.arange(k)]).astype(np.int32)
    return gen.EdgeList(n=g.n + k, src=np.concatenate([g.src, t[:-1]]), dst=np.concatenate([g.dst, t[1:]]))


DEEP_CASES = {
    "grid-w": gen.with_weights(gen.grid(60, 60), 16, seed=41),        # given up early
    "tail-past": gen.with_weights(with_tail(gen.erdos_renyi(600, 0.01, seed=42), 90), 9, seed=42),   # at the last level
    "tail-within": gen.with_weights(with_tail(gen.erdos_renyi(600, 0.01, seed=43), 25), 9, seed=43),
    "islands-w": gen.with_weights(union(gen.erdos_renyi(300, 0.03, seed=44), gen.path(60), gen.star(50)), 5, seed=44),
    "cycle": gen.cycle(150),
}


@pytest.mark.parametrize("name", list(DEEP_CASES))
def test_deep_graphs(bc, name):
    """Calls without a bound on the levels, around the test for a deep graph at a quarter of them."""
    g = DEEP_CASES[name]
    S = gen.sample_targets(g.n, 45, seed=3)
    ref, _ = oracle.brandes(g, S)
    got = bc.brandes(bc.graph_from_edgelist(g), S, order_sources=False).cpu().numpy()
    assert rel_err(got, ref) <= FP64_TOL


def test_deep_graphs_batched(bc):
    gs = [gen.erdos_renyi(80, 0.06, seed=45), gen.cycle(140), gen.grid(3, 50), gen.path(120)]
    arena = bc.build_arena(gs)
    got = bc.brandes_batched(arena).cpu().numpy()
    for i, g in enumerate(gs):
        ref, _ = oracle.brandes(g, None)
        assert rel_err(got[arena.node_ptr_host[i]:arena.node_ptr_host[i + 1]], ref) <= FP64_TOL, i


@pytest.mark.parametrize("rungs", [97, 98, 99, 140])
@pytest.mark.parametrize("every", [1, 4, 5])
def test_long_graphs_by_density_of_targets(bc, rungs, every):
    """A ladder around the depth past which calls with many targets run on the lockstep kernel."""
    g = gen.grid(2, rungs)
    S = np.arange(0, g.n, every, dtype=np.int32)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    assert rel_err(bc.brandes(G, S).cpu().numpy(), ref) <= FP64_TOL
    part = (np.arange(g.n) % rungs // 10).astype(np.int32)
    assert rel_err(bc.brandes_pp(G, S, part).cpu().numpy(), ref) <= FP64_TOL
