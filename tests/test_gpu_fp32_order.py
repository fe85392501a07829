"""GPU: FP32 dependencies on the level-mask kernel are added in the lockstep kernel's order.  The same graph with a
weight of one on every edge takes the lockstep kernel with the same batches: the FP32 values are the same bits, so
the results agree to the rounding of their FP64 sums (another order of FP32 additions differs in the 7th or 8th digit)."""
import numpy as np
import pytest

from paper_1406_4173_gb300 import api, gen

pytestmark = pytest.mark.gpu

# sums over sources in FP64: at most a few hundred terms, each order within 2^-53 per term of the exact sum
SUM_TOL = 1e-12


@pytest.fixture(scope="module")
def bc():
    import torch
    import paper_1406_4173_gb300 as m
    from paper_1406_4173_gb300 import _build
    _build.build()
    torch.cuda.set_device(0)
    return m


def hub_over(deg, seed):
    """A hub over a sparse random graph of its neighbours: rows of more than 256 arcs."""
    g = gen.erdos_renyi(deg, min(1.0, 4.0 / deg), seed=seed)
    return gen.EdgeList(n=deg + 1, src=np.concatenate([np.zeros(deg, np.int32), g.src + 1]).astype(np.int32),
                        dst=np.concatenate([np.arange(1, deg + 1), g.dst + 1]).astype(np.int32))


def ones(g):
    return gen.EdgeList(n=g.n, src=g.src, dst=g.dst, w=np.ones(len(g.src), np.uint32), directed=g.directed)


CASES = {
    **{f"hub{d}": hub_over(d, d) for d in (200, 255, 256, 257, 300, 513, 1025)},
    "star": gen.star(700),                 # up to 31 sources of a batch at one distance
    "complete": gen.complete(90),
    "random": gen.erdos_renyi(900, 0.01, seed=7),
    "planted": gen.planted_partition(800, 8, 0.05, 0.004, seed=8),
    "directed": gen.chung_lu_communities(900, [180] * 5, 2.2, 8.0, 0.85, seed=9, directed=True),
}


def rel(x, y):
    return float(np.max(np.abs(x - y) / np.maximum(np.abs(y), 1.0)))


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("k", [1, 7, 32, 33, None])
def test_same_bits_as_lockstep(bc, name, k):
    g = CASES[name]
    S = None if k is None else gen.sample_targets(g.n, max(2, k), seed=3)
    ctx = bc.Context()
    out = []
    for x, kernel in ((g, "levels"), (ones(g), "lockstep")):
        out.append(bc.brandes(bc.graph_from_edgelist(x), S, precision="fp32", order_sources=False, ctx=ctx).cpu().numpy())
        b = ctx.last_batches()
        assert b[kernel] > 0 and sum(b.values()) == b[kernel]
    ctx.close()
    assert rel(*out) <= SUM_TOL


def test_same_bits_as_lockstep_batched(bc):
    gs = [CASES[n] for n in ("hub257", "star", "complete", "random", "planted")] + [gen.erdos_renyi(33, 0.2, seed=1)]
    arena = bc.build_arena(gs)
    off = np.repeat(arena.node_ptr_host[:-1], [len(g.src) for g in gs])
    src, dst = (np.concatenate([getattr(g, e) for g in gs]) + off for e in ("src", "dst"))
    G = bc.csr_build(int(arena.node_ptr_host[-1]), src.astype(np.int32), dst.astype(np.int32),
                     np.ones(len(src), np.uint32), False)
    ctx = bc.Context()
    out = []
    for x, kernel in ((arena, "levels"), (api.Arena(arena.node_ptr, arena.node_ptr_host, G), "lockstep")):
        out.append(bc.brandes_batched(x, precision="fp32", ctx=ctx).cpu().numpy())
        assert ctx.last_batches()[kernel] > 0 and ctx.last_batches()["given_back"] == 0
    ctx.close()
    assert rel(*out) <= SUM_TOL
