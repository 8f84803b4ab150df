"""The peel's bands (levels grouped by one cascade, then peeled side by side)
and the one-block h = 2 peel, at the sizes where their bookkeeping changes."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1906_00341_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1906_00341_gb300 import build as b
    b.build()
    from paper_1906_00341_gb300 import _lib
    _lib.load()
    return _lib


def ring(n, w, drop, seed):
    """Ring lattice (neighbours at distance <= w) with a share of its edges gone:
    a cascade that starts at a defect runs around the whole ring."""
    i = np.arange(n, dtype=np.int64)
    s = np.concatenate([i] * w)
    d = np.concatenate([(i + j) % n for j in range(1, w + 1)])
    keep = np.random.default_rng(seed).random(s.size) >= drop
    return n, s[keep].astype(np.uint32), d[keep].astype(np.uint32)


@pytest.mark.parametrize("limit", [0, 300, 1 << 30])
@pytest.mark.parametrize("h", [2, 3, 4])
def test_band_cascades(L, orc, h, limit):
    """Cascades above the band limit (undone, the level taken alone), bands of
    every size on a power-law graph, and no bands at all: core numbers, level
    records and mu equal the oracle's."""
    graphs = [ring(30000, 4, 0.002, 1),
              gg.plant(20000, *gg.chung_lu(20000, 160000, 2.1, 900.0, 5)[1:], 70, 0.6, 6)[:3]]
    L.dsd_set_peel_tail_limit(limit)
    try:
        for n, s, d in graphs:
            og = orc.csr(n, s, d)
            wcore, wk = orc.core_decompose(og, h)
            wl = orc.level_stats(og, h, wcore)
            with L.Graph.from_edges(n, s, d) as g:
                core, k = g.core_decompose(h)
                lv = g.level_stats(h)
            assert k == wk and np.array_equal(core, wcore)
            for a, b in zip(lv, wl):
                assert np.array_equal(np.asarray(a, np.uint64), np.asarray(b, np.uint64))
    finally:
        L.dsd_set_peel_tail_limit(1 << 30)


def rounds_of(n, s, d):
    """Core numbers and removal rounds of the level-synchronous h = 2 peel."""
    lo, hi = np.minimum(s, d).astype(np.int64), np.maximum(s, d).astype(np.int64)
    key = np.unique((lo * n + hi)[lo != hi])
    u, v = key // n, key % n
    src, dst = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.argsort(src, kind="stable")
    src, dst = src[order], dst[order]
    off = np.searchsorted(src, np.arange(n + 1))
    deg = np.diff(off)
    core, rnd = np.zeros(n, np.int64), np.zeros(n, np.int64)
    alive = np.ones(n, bool)
    k = r = 0
    while alive.any():
        k = max(k, int(deg[alive].min()))
        f = np.nonzero(alive & (deg <= k))[0]
        while f.size:
            core[f], rnd[f], alive[f] = k, r, False
            nb = np.concatenate([dst[off[x]:off[x + 1]] for x in f])
            np.subtract.at(deg, nb, 1)
            f = np.nonzero(alive & (deg <= k))[0]
            r += 1
    return core, rnd


@pytest.mark.parametrize("n,m", [(1, 0), (33, 60), (1025, 5000), (16384, 60000), (16385, 60000),
                                 (3000, 199900), (3000, 240000)])
def test_one_block_order(L, n, m):
    """h = 2 on both sides of the one-block limits: core numbers and the order
    by (removal round, id)."""
    if m:
        n, s, d = gg.chung_lu(n, m, 2.3, 4.0 * n ** 0.5, n)
    else:
        s = d = np.zeros(0, np.uint32)
    core, rnd = rounds_of(n, s, d)
    rank = np.empty(n, np.int64)
    rank[np.lexsort((np.arange(n), rnd))] = np.arange(n)
    with L.Graph.from_edges(n, s, d) as g:
        c2, rk, _ = g.degeneracy_order()
    assert np.array_equal(c2, core)
    assert np.array_equal(rk, rank)


@pytest.mark.parametrize("x", [2, 3, 5])
@pytest.mark.parametrize("graph", ["ring", "power", "dense", "hub"])
def test_star_bands(L, graph, x):
    """The x-star peel in bands against the one-level peel (limit 0, itself
    compared with the oracle in the pattern tests): a cascade around a ring
    (undone), a power law, one dense block, and a hub whose counts may pass
    2^62 (x = 5: C(40000, 5) > 2^62, not taken in bands)."""
    if graph == "ring":
        n, s, d = ring(20000, 3, 0.003, 2)
    elif graph == "power":
        n, s, d = gg.chung_lu(9001, 70000, 2.1, 700.0, 3)
        s, d = np.concatenate([s, [0, 8999]]).astype(np.uint32), \
            np.concatenate([d, [9000, 9000]]).astype(np.uint32)
    elif graph == "dense":
        n, s, d = gg.er(700, 0.2, 4)
    else:
        n, s, d = gg.er(40001, 0.00002, 5)
        s = np.concatenate([s, np.zeros(40000, np.uint32)])
        d = np.concatenate([d, np.arange(1, 40001, dtype=np.uint32)])
    got = []
    with L.Graph.from_edges(n, s, d) as g:
        for limit in (0, 500, 1 << 30):
            L.dsd_set_peel_tail_limit(limit)
            try:
                got.append(g.pattern_core_decompose(L.DSD_PATTERN_STAR, x))
            finally:
                L.dsd_set_peel_tail_limit(1 << 30)
    for r in got[1:]:
        assert r[1] == got[0][1]
        for a, b in zip(r, got[0]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("case", ["n3072", "n3073", "m16384", "m16385", "row256", "row257",
                                  "row3000", "repeats", "bad"])
def test_one_block_csr(L, orc, case):
    """The one-block CSR build and orientation on both sides of their limits, a
    row beyond the block's buffer through repeats, and a bad endpoint."""
    rng = np.random.default_rng(7)
    if case[0] == "n":
        n, m = int(case[1:]), 12000
        s, d = rng.integers(0, n, m), rng.integers(0, n, m)
    elif case[0] == "m":
        n, m = 3000, int(case[1:])
        s, d = rng.integers(0, n, m), rng.integers(0, n, m)
    elif case == "repeats":
        n, m = 300, 16000
        s, d = np.zeros(m, np.int64), rng.integers(0, n, m)
    elif case == "bad":
        with pytest.raises(L.DSDError) as ei:
            L.Graph.from_edges(100, np.array([0, 5, 100], np.uint32),
                               np.array([1, 6, 2], np.uint32))
        assert ei.value.name == "DSD_ERR_INVALID"
        return
    else:
        k = int(case[3:])
        n = k + 50
        s = np.concatenate([np.zeros(k, np.int64), rng.integers(0, n, 2 * k)])
        d = np.concatenate([np.arange(1, k + 1), rng.integers(0, n, 2 * k)])
    s, d = s.astype(np.uint32), d.astype(np.uint32)
    og = orc.csr(n, s, d)
    core, rnd = rounds_of(n, s, d)
    rank = np.empty(n, np.int64)
    rank[np.lexsort((np.arange(n), rnd))] = np.arange(n)
    with L.Graph.from_edges(n, s, d) as g:
        off, adj = g.csr()
        c2, rk, _ = g.degeneracy_order()
        deg, mu = g.clique_degrees(3)
    assert np.array_equal(off, og.off) and np.array_equal(adj, og.adj)
    assert np.array_equal(c2, core) and np.array_equal(rk, rank)
    wdeg, wmu = orc.clique_degrees(og, 3)
    assert mu == wmu and np.array_equal(deg, wdeg)


def test_release_memory(L):
    """The library's pool keeps at most 2 GiB and gives it back on request."""
    import torch
    L.dsd_release_memory()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    n, s, d = gg.er(200_000, 0.0002, 3)
    for _ in range(2):
        with L.Graph.from_edges(n, s, d) as g:
            g.core_app(3)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free0 - (2 << 30) - (64 << 20)
    L.dsd_release_memory()
    assert torch.cuda.mem_get_info()[0] >= free0 - (64 << 20)
