"""GPU: Brandes++ with little device memory left.  Centrality's frontier lists are sized before the batches'
workspace, and where they would take most of what is left it reads the Dijkstra_SK tables instead."""
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


def ring_of_parts(k, size, ends, directed, seed):
    """k random parts of mean degree 10; `ends` random nodes of each tied to the next part."""
    r = np.random.default_rng(seed)
    src, dst = [], []
    for i in range(k):
        u = r.integers(0, size, 5 * size)
        v = (u + r.integers(1, size, 5 * size)) % size
        src += [u + i * size, r.choice(size, ends, replace=False) + i * size]
        dst += [v + i * size, r.choice(size, ends, replace=False) + (i + 1) % k * size]
    s, d = np.concatenate(src), np.concatenate(dst)
    if directed:
        s, d = np.concatenate([s, d[::2]]), np.concatenate([d, s[::2]])
    else:
        s, d = np.minimum(s, d), np.maximum(s, d)
    key = np.unique(s.astype(np.int64) * (k * size) + d)
    return gen.EdgeList(n=k * size, src=(key // (k * size)).astype(np.int32), dst=(key % (k * size)).astype(np.int32),
                        part=(np.arange(k * size) // size).astype(np.int32), directed=directed)


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_centrality_without_lists(bc, directed, precision):
    """24 million table entries, nearly all of them listed: 384 MB of lists (directed: of each kind)."""
    import torch
    g = ring_of_parts(4, 10000, 300, directed, seed=5)
    S = gen.sample_targets(g.n, 40, seed=3)
    ref, _ = oracle.brandes(g, S)
    G = bc.graph_from_edgelist(g)
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - ((1500 if directed else 900) << 20), dtype=torch.uint8, device="cuda")
    ctx = bc.Context()
    try:
        x, st = bc.brandes_pp(G, S, g.part, precision=precision, stats=True, ctx=ctx)
        x = x.cpu().numpy()
    finally:
        ctx.close()
        del hold
        torch.cuda.empty_cache()
    assert st["table_entries"] > 20e6
    err = float(np.max(np.abs(x - ref) / np.maximum(np.abs(ref), 1.0)))
    assert err <= (FP64_TOL if precision == "fp64" else 2e-6)
