"""GPU: bcpp_csr_build against a host sort, with row lengths around its sorting classes (a warp's 32
registers, 512 in a warp's shared memory, the powers of two of the block sort, the whole-graph sort
above 16,384), directed and undirected, with and without weights, edges in random order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bc():
    import torch
    import paper_1406_4173_gb300 as m
    from paper_1406_4173_gb300 import _build
    _build.build()
    torch.cuda.set_device(0)
    return m


def host_csr(n, src, dst, w, directed):
    u = src if directed else np.concatenate([src, dst])
    v = dst if directed else np.concatenate([dst, src])
    x = w if directed else np.concatenate([w, w])
    o = np.lexsort((v, u))
    rp = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=n))])
    return rp, v[o], x[o]


@pytest.mark.parametrize("deg", [1, 2, 31, 32, 33, 64, 65, 255, 256, 257, 511, 512, 513, 1024, 4000, 16384, 16385])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("weighted", [False, True])
def test_build_matches_host_sort(bc, deg, directed, weighted):
    rng = np.random.default_rng(deg)
    n = deg + 7
    hub = 3
    heads = rng.permutation(np.delete(np.arange(n), hub))[:deg]
    keys = [hub * n + heads] if directed else [np.minimum(hub, heads) * n + np.maximum(hub, heads)]
    u, v = rng.integers(0, n, 4 * min(n, 500)), rng.integers(0, n, 4 * min(n, 500))
    ok = (u != v) & (u != hub) & (v != hub)
    u, v = u[ok], v[ok]
    keys.append(u * n + v if directed else np.minimum(u, v) * n + np.maximum(u, v))
    k = rng.permutation(np.unique(np.concatenate(keys)))
    src, dst = (k // n).astype(np.int32), (k % n).astype(np.int32)
    w = rng.integers(1, 1000, k.size).astype(np.uint32)
    G = bc.csr_build(n, src, dst, w if weighted else None, directed)
    rp, col, wo = host_csr(n, src, dst, w, directed)
    assert np.array_equal(G.row_ptr.cpu().numpy(), rp)
    assert np.array_equal(G.col.cpu().numpy(), col)
    if weighted:
        assert np.array_equal(G.w.cpu().numpy().view(np.uint32), wo)


@pytest.mark.parametrize("deg", [5, 40, 300, 600, 20000])
@pytest.mark.parametrize("what", ["repeat", "repeat-other-weight", "loop", "range", "zero-weight"])
def test_build_refuses(bc, deg, what):
    n = deg + 2
    src, dst = np.zeros(deg, np.int32), np.arange(1, deg + 1, dtype=np.int32)
    w = np.ones(deg, np.uint32)
    if what.startswith("repeat"):
        dst[-1] = dst[0]
        w[-1] = 7 if "other" in what else 1
    elif what == "loop":
        dst[-1] = 0
    elif what == "range":
        dst[-1] = n
    else:
        w[-1] = 0
    for directed in (False, True):
        with pytest.raises(bc.BcppError):
            bc.csr_build(n, src, dst, w, directed)


@pytest.mark.parametrize("a", [0, 1, 2, 3, 8, 9, 15, 16, 17, 32, 33])
@pytest.mark.parametrize("b", [0, 1, 5, 16, 17])
@pytest.mark.parametrize("weighted", [False, True])
def test_build_pairs_of_rows(bc, a, b, weighted):
    """Two rows to a warp: lengths a and b side by side, an odd number of rows, one repeated head at a time."""
    rng = np.random.default_rng(100 * a + b)
    n = 41
    src = np.concatenate([np.full(a if u % 2 == 0 else b, u) for u in range(n)]).astype(np.int32)
    dst = np.concatenate([rng.choice(np.delete(np.arange(n), u), a if u % 2 == 0 else b, replace=False)
                          for u in range(n)]).astype(np.int32)
    o = rng.permutation(src.size)
    src, dst = src[o], dst[o]
    w = rng.integers(1, 1000, src.size).astype(np.uint32)
    G = bc.csr_build(n, src, dst, w if weighted else None, True)
    rp, col, wo = host_csr(n, src, dst, w, True)
    assert np.array_equal(G.row_ptr.cpu().numpy(), rp)
    assert np.array_equal(G.col.cpu().numpy(), col)
    if weighted:
        assert np.array_equal(G.w.cpu().numpy().view(np.uint32), wo)
    for u in (0, 1):
        at = np.nonzero(src == u)[0]
        if at.size:
            with pytest.raises(bc.BcppError):
                bc.csr_build(n, np.append(src, np.int32(u)), np.append(dst, dst[at[0]]),
                             np.append(w, np.uint32(7)) if weighted else None, True)


@pytest.mark.parametrize("hubs", [1, 2, 5])
@pytest.mark.parametrize("end", ["first", "second"])
@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("weighted", [False, True])
def test_build_several_long_rows(bc, hubs, end, shuffled, directed, weighted):
    """Rows above 16,384 arcs are sorted apart: several of them, with shorter rows between, their nodes as first or
    second ends, grouped (a warp's edges share an end) or not."""
    rng = np.random.default_rng(hubs)
    n, deg = 20011, 16384 + 37
    ids = np.sort(rng.choice(n, hubs, replace=False))
    pairs = [np.stack([np.full(deg, h), rng.choice(np.delete(np.arange(n), ids), deg, replace=False)]) for h in ids]
    pairs.append(rng.choice(np.delete(np.arange(n), ids), (2, 3000)))
    a, b = np.concatenate(pairs, axis=1)
    if end == "second":
        a, b = b, a
    key = np.minimum(a, b).astype(np.int64) * n + np.maximum(a, b)
    keep = np.unique(key, return_index=True)[1]
    keep = keep[a[keep] != b[keep]]
    keep = rng.permutation(keep) if shuffled else np.sort(keep)
    src, dst = a[keep].astype(np.int32), b[keep].astype(np.int32)
    w = rng.integers(1, 1000, len(src)).astype(np.uint32)
    G = bc.csr_build(n, src, dst, w if weighted else None, directed)
    rp, col, ww = host_csr(n, src, dst, w, directed)
    assert np.array_equal(G.row_ptr.cpu().numpy(), rp)
    assert np.array_equal(G.col.cpu().numpy(), col)
    if weighted:
        assert np.array_equal(G.w.cpu().numpy().view(np.uint32), ww)


def test_build_of_nothing(bc):
    none = np.zeros(0, np.int32)
    for n in (0, 1, 70):
        G = bc.csr_build(n, none, none, None, False)
        assert np.array_equal(G.row_ptr.cpu().numpy(), np.zeros(n + 1, np.int64)) and G.col.numel() == 0
