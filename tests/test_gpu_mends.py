"""Calls that earlier forms of the kernels answered wrongly, refused or slowed
down, each at the smallest input that shows it."""
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


def clique(v):
    v = np.asarray(v, np.int64)
    i, j = np.triu_indices(v.size, 1)
    return v[i], v[j]


def late_member():
    """h = 5: an item (v, w) whose first 128 entries of N+(w) hold more than
    four members of later bands and only then x, which is in v's band.

    Ids 0-9 are W, a clique with v and x (so v has C(11, 4) = 330 cliques) and
    with 10 more vertices Z (a later band); each of W has 150 further
    neighbours among Q, which lie between W and x in the degeneracy order: Q
    is one side of a complete bipartite graph (no triangles there) and x is of
    the other side.  x is in 35 cliques of a K13 besides.  400 disjoint K14,
    one vertex of each next to v, keep v's row long.  K5, K6 and K7 give v's
    band its first levels."""
    W = np.arange(10)
    at = [10]

    def take(k):
        at[0] += k
        return np.arange(at[0] - k, at[0])
    v, = take(1)
    Z = take(10)
    Q = take(1500)
    P = take(220)
    x = P[0]
    E = [clique(np.concatenate([W, [v, x]])), clique(np.concatenate([W, Z]))]
    E.append((np.repeat(P, Q.size), np.tile(Q, P.size)))
    E += [(np.full(150, w), Q[150 * w:150 * w + 150]) for w in W]
    k13 = take(13)
    E += [clique(k13), (np.full(7, x), k13[:7])]
    for _ in range(400):
        c = take(14)
        E += [clique(c), (np.array([v]), c[:1])]
    E += [clique(take(k)) for k in (5, 6, 7)]
    return (at[0], np.concatenate([a for a, _ in E]).astype(np.uint32),
            np.concatenate([b for _, b in E]).astype(np.uint32), v, x)


@pytest.mark.parametrize("warp_max", [4, 16, 32])
def test_queue_off_long_rows(L, orc, warp_max):
    """dsd_set_peel_items(w, 0): a candidate walk that stops at w candidates says
    nothing about the rest of the row, so its item must reach a block."""
    n, s, d, v, x = late_member()
    og = orc.csr(n, s, d)
    wcore, wk = orc.core_decompose(og, 5)
    wl = orc.level_stats(og, 5, wcore)
    assert wcore[v] == wcore[x] == 330
    L.dsd_set_peel_items(warp_max, 0)
    try:
        with L.Graph.from_edges(n, s, d) as g:
            core, k = g.core_decompose(5)
            lv = g.level_stats(5)
    finally:
        L.dsd_set_peel_items(4, 1 << 20)
    assert k == wk and np.array_equal(core, wcore)
    for a, b in zip(lv, wl):
        assert np.array_equal(np.asarray(a, np.uint64), np.asarray(b, np.uint64))


def test_star_without_room(L):
    """The x-star peel on a device with room for the one-level peel but not for
    the bands' 56 bytes an edge (20M edges): the same result, no error."""
    import torch
    n, w = 1_000_000, 20
    i = np.arange(n, dtype=np.int64)
    s = np.tile(i, w).astype(np.uint32)
    d = np.concatenate([(i + j) % n for j in range(1, w + 1)]).astype(np.uint32)
    with L.Graph.from_edges(n, s, d) as g:
        want = g.pattern_core_decompose(L.DSD_PATTERN_STAR, 2)
        L.dsd_release_memory()
        torch.cuda.synchronize()
        hold = torch.empty(torch.cuda.mem_get_info()[0] - (600 << 20), dtype=torch.uint8,
                           device="cuda")
        try:
            got = g.pattern_core_decompose(L.DSD_PATTERN_STAR, 2)
        finally:
            del hold
            torch.cuda.empty_cache()
    assert got[1] == want[1] == 780 + 40 * 39   # C(40, 2) + 40 C(39, 1) at every vertex
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("keep", [0, 64 << 20])
def test_memory_keep(L, keep):
    """dsd_set_memory_keep: after a synchronisation no more than the bound of
    freed memory stays with the library (the default keeps up to 2 GiB, which
    another allocator of the process could not have)."""
    import torch
    L.dsd_release_memory()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    n, s, d = gg.er(200_000, 0.0002, 3)   # 4M edges: some 500 MB in use at a time
    L.dsd_set_memory_keep(keep)
    try:
        for _ in range(2):
            with L.Graph.from_edges(n, s, d) as g:
                g.core_app(3)
            torch.cuda.synchronize()
            assert torch.cuda.mem_get_info()[0] >= free0 - keep - (64 << 20)
    finally:
        L.dsd_set_memory_keep(2 << 30)
        L.dsd_release_memory()


def test_peel_stats_names(L):
    """Every word of dsd_peel_stats under the name of what it holds: the 100
    levels of a K3 .. K102 each (h = 2) in bands, and none with bands off."""
    sizes = range(3, 103)
    base = np.cumsum([0] + [k for k in sizes])
    E = [clique(b + np.arange(k)) for b, k in zip(base, sizes)]
    n = int(base[-1]) + 20_000   # vertices without edges: not one block's graph
    s = np.concatenate([a for a, _ in E]).astype(np.uint32)
    d = np.concatenate([b for _, b in E]).astype(np.uint32)
    for limit in (1 << 30, 0):
        L.dsd_set_peel_tail_limit(limit)
        try:
            with L.Graph.from_edges(n, s, d) as g:
                g.core_app(3)
                st = L.dsd_peel_stats(g.handle, 1)
        finally:
            L.dsd_set_peel_tail_limit(1 << 30)
        assert st["levels"] == 101 and st["kmax"] == 101 * 100 // 2
        if limit:
            # bands of more than one level, all begun on the 5,250 vertices left
            # after level 0 or before it; fewer grid rounds than rounds
            assert 1 <= st["bands"] <= 50 and 0 < st["band_n"] <= n
            assert 0 < st["phase2_ns"] < 10 ** 10
            assert st["grid_rounds"] < st["rounds"]
        else:
            assert st["bands"] == st["band_n"] == st["phase2_ns"] == 0
            assert st["grid_rounds"] == st["rounds"]


@pytest.mark.parametrize("n,p", [(2000, 0.005), (40_000, 0.0005)])
def test_phase_launches(L, n, p):
    """The kernels dsd_phase_stats says each phase launched, against the
    library's own count: one-block stages and the general ones."""
    n, s, d = gg.er(n, p, 1)
    at = [L.dsd_kernel_launches()]
    with L.Graph.from_edges(n, s, d) as g:
        at.append(L.dsd_kernel_launches())
        g.degeneracy_order()
        at.append(L.dsd_kernel_launches())
        g.clique_degrees(3)
        at.append(L.dsd_kernel_launches())
        csr, peel, orient, count = [int(x) for x in L.dsd_phase_stats(g.handle)[2][:4]]
    assert min(csr, peel, orient, count) > 0
    assert csr == at[1] - at[0]
    assert peel + orient <= at[2] - at[1] <= peel + orient + 1   # and the core numbers' map
    assert count <= at[3] - at[2] <= count + 1                   # and the counts'


def test_band_aim(L):
    """However many vertices are alive, a band's threshold is set for at most
    2,048 of them: 4M vertices in K6 (10 triangles each), 1,800 in single
    triangles and 600 in K4 (3 each) make no band of several levels."""
    def many(k, count, at):
        i, j = np.triu_indices(k, 1)
        o = at + k * np.arange(count)[:, None]
        return (o + i).ravel(), (o + j).ravel(), at + k * count
    s6, d6, at = many(6, 666_700, 0)
    s3, d3, at = many(3, 600, at)
    s4, d4, n = many(4, 150, at)
    s = np.concatenate([s6, s3, s4]).astype(np.uint32)
    d = np.concatenate([d6, d3, d4]).astype(np.uint32)
    with L.Graph.from_edges(n, s, d) as g:
        core, k = g.core_decompose(3)
        lk, ls, lm = g.level_stats(3)
        st = L.dsd_peel_stats(g.handle, 1)
    assert k == 10 and np.array_equal(lk, [1, 3, 10])
    assert np.array_equal(ls, [n, n - 1800, n - 2400])
    assert np.array_equal(lm, [20 * 666_700 + 600 + 4 * 150, 20 * 666_700 + 4 * 150, 20 * 666_700])
    assert np.array_equal(core, np.repeat([10, 1, 3], [6 * 666_700, 1800, 600]))
    assert st["bands"] == 0


def strip(n, w):
    """Vertices in a row, each next to the w before and after it: one level that
    leaves from the two ends, a vertex each a round."""
    i = np.arange(n, dtype=np.int64)
    s = np.concatenate([i[:n - j] for j in range(1, w + 1)])
    d = np.concatenate([i[j:] for j in range(1, w + 1)])
    return n, s.astype(np.uint32), d.astype(np.uint32)


@pytest.mark.parametrize("n,h", [(3000, 3), (3000, 5), (7000, 4), (40_000, 2)])
def test_long_cascade(L, orc, n, h):
    """A cascade along a path is not run twice (as a band and again level by
    level): 48 rounds a try at most on top of the peel's own."""
    n, s, d = strip(n, max(h - 1, 1))
    og = orc.csr(n, s, d)
    wcore, wk = orc.core_decompose(og, h)
    wl = orc.level_stats(og, h, wcore)
    with L.Graph.from_edges(n, s, d) as g:
        core, k = g.core_decompose(h)
        lv = g.level_stats(h)
        st = L.dsd_peel_stats(g.handle, 0 if h == 2 else 1)
    assert k == wk and np.array_equal(core, wcore)
    for a, b in zip(lv, wl):
        assert np.array_equal(np.asarray(a, np.uint64), np.asarray(b, np.uint64))
    assert st["rounds"] >= n // 2 - 8
    assert st["grid_rounds"] <= st["rounds"] + 4 * 48


@pytest.mark.parametrize("x", [2, 3])
@pytest.mark.parametrize("graph", ["strips", "path", "er", "power"])
def test_star_long_cascade(L, graph, x):
    """A round of the x-star peel that changes little costs little: 2,000 strips of
    400 vertices (200 rounds; gathered anew each round it took 5.6 times the
    one-level peel).  The other graphs mix rounds passed on as differences with
    gathered ones; all equal the one-level peel."""
    import time
    if graph == "strips":
        _, s1, d1 = strip(400, 2)
        at = 400 * np.arange(2000)[:, None]
        n, s, d = 800_000, (s1 + at).ravel().astype(np.uint32), (d1 + at).ravel().astype(np.uint32)
    elif graph == "path":
        n, s, d = strip(9000, 1)
    elif graph == "er":
        n, s, d = gg.er(60_000, 0.0001, 4)
    else:
        n, s, d = gg.chung_lu(20_000, 160_000, 2.1, 900.0, 5)
    best = {}
    got = {}
    with L.Graph.from_edges(n, s, d) as g:
        for limit in (0, 1 << 30):
            L.dsd_set_peel_tail_limit(limit)
            try:
                for _ in range(3):
                    t = time.perf_counter()
                    got[limit] = g.pattern_core_decompose(L.DSD_PATTERN_STAR, x)
                    t = time.perf_counter() - t
                    best[limit] = min(best.get(limit, t), t)
            finally:
                L.dsd_set_peel_tail_limit(1 << 30)
    for a, b in zip(got[0], got[1 << 30]):
        assert np.array_equal(a, b)
    if graph == "strips":
        assert best[1 << 30] < 2 * best[0]


@pytest.mark.parametrize("h,w,count,length", [
    (3, 2, 1, 3000),     # a vertex at each end a round
    (3, 2, 32, 300),     # 64 vertices a round: one block's
    (3, 2, 33, 300),     # 66: the grid's
    (4, 8, 3, 500),      # rows of 16
    (4, 9, 3, 500),      # rows of 18
    (5, 4, 2, 900), (6, 5, 1, 700), (3, 2, 1, 9)])
def test_narrow_rounds(L, orc, h, w, count, length):
    """Rounds of a few vertices with short rows run in one block (they took two
    grid barriers each), on both sides of its limits and beside a larger graph
    whose rounds are the grid's."""
    _, s1, d1 = strip(length, w)
    at = length * np.arange(count)[:, None]
    n = length * count
    _, se, de = gg.er(500, 0.1, 3)
    s = np.concatenate([(s1 + at).ravel(), se + n]).astype(np.uint32)
    d = np.concatenate([(d1 + at).ravel(), de + n]).astype(np.uint32)
    for nn, m in ((n, count * s1.size), (n + 500, s.size)):
        og = orc.csr(nn, s[:m], d[:m])
        wcore, wk = orc.core_decompose(og, h)
        wl = orc.level_stats(og, h, wcore)
        for limit in (1 << 30, 0):
            L.dsd_set_peel_tail_limit(limit)
            try:
                with L.Graph.from_edges(nn, s[:m], d[:m]) as g:
                    core, k = g.core_decompose(h)
                    lv = g.level_stats(h)
                    st = L.dsd_peel_stats(g.handle, 1)
            finally:
                L.dsd_set_peel_tail_limit(1 << 30)
            assert k == wk and np.array_equal(core, wcore)
            for a, b in zip(lv, wl):
                assert np.array_equal(np.asarray(a, np.uint64), np.asarray(b, np.uint64))
            if nn == n and 2 * count <= 64 and 2 * w <= 16 and length > 100 and limit == 0:
                assert st["barriers"] < st["rounds"] // 2 + 20


@pytest.mark.parametrize("kind", ["empty", "sparse", "one_large"])
def test_batch_more_vertices_than_entries(L, orc, kind):
    """A batch whose largest graph has more vertices than any has row entries:
    the (round, id) keys have room (they ran over the rows behind them)."""
    e = np.zeros(0, np.uint32)
    rng = np.random.default_rng(5)
    if kind == "empty":
        graphs = [(100, e, e, 2 + i % 3) for i in range(9)] + [(1, e, e, 3), (65535, e, e, 4)]
    elif kind == "sparse":
        graphs = []
        for i in range(12):
            n, k = 300 + 117 * i, 6 + i
            at = rng.choice(n, k, replace=False).astype(np.uint32)
            a, b = np.triu_indices(k, 1)
            graphs.append((n, at[a], at[b], 2 + i % 3))
    else:
        _, s, d = gg.er(120, 0.2, 1)
        graphs = [(120, s, d, h) for h in (2, 3, 4)]
        graphs += [(60_000, np.array([7, 7, 9], np.uint32), np.array([9, 59_999, 59_999], np.uint32), h)
                   for h in (3, 4)]
    b = L.Batch(graphs, want_cores=True)
    b.run()
    res = b.results()
    for (n, s, d, h), r in zip(graphs, res):
        og = orc.csr(n, s, d)
        core, k = orc.core_decompose(og, h)
        assert r["status"] == 0 and r["kmax"] == k and np.array_equal(r["core"], core)
    b.close()


@pytest.mark.parametrize("rows,length,general", [(50, 300, True), (3, 300, False),
                                                 (20, 1600, True), (1, 3000, False),
                                                 (16, 1000, False), (17, 1000, True)])
def test_small_csr_long_rows(L, orc, rows, length, general):
    """The one-block CSR build leaves graphs with many long rows, which it sorts
    one after another, to the general path (more than its one launch)."""
    rng = np.random.default_rng(rows)
    n = 3050
    s = np.repeat(np.arange(rows), length)
    d = np.concatenate([rows + rng.permutation(n - rows)[:length] if length < 1600 or rows == 1
                        else rng.integers(rows, n, length) for _ in range(rows)])
    keep = rng.permutation(s.size)[:16384]
    s, d = s[keep].astype(np.uint32), d[keep].astype(np.uint32)
    og = orc.csr(n, s, d)
    with L.Graph.from_edges(n, s, d) as g:
        off, adj = g.csr()
        launches = int(L.dsd_phase_stats(g.handle)[2][0])
        core, _, _ = g.degeneracy_order()
    assert np.array_equal(off, og.off) and np.array_equal(adj, og.adj)
    wcore, _ = orc.core_decompose(og, 2)
    assert np.array_equal(core, wcore)
    assert (launches > 1) == general


def test_batch_long_rows(L, orc):
    """The batch kernel's frontiers: many vertices with rows on both sides of
    128 entries (a warp each, or listed and shared by the block), few vertices
    (shared) and hubs beside short rows."""
    graphs = []
    for h in (2, 3, 4):
        graphs += [(400, *gg.er(400, 0.32, h)[1:], h), (300, *gg.er(300, 0.6, h)[1:], h),
                   (*strip(700, 3), h)]
        _, s, d = gg.er(900, 0.02, h)
        hub = np.arange(1, 900, dtype=np.uint32)
        graphs.append((900, np.concatenate([s, np.zeros(899, np.uint32)]),
                       np.concatenate([d, hub]), h))
    b = L.Batch(graphs, want_cores=True)
    b.run()
    for (n, s, d, h), r in zip(graphs, b.results()):
        og = orc.csr(n, s, d)
        core, k = orc.core_decompose(og, h)
        lk, ls, lm = orc.level_stats(og, h, core)
        assert r["status"] == 0 and r["kmax"] == k and np.array_equal(r["core"], core)
        assert r["nlevels"] == len(lk) and r["kmax_core_size"] == ls[-1]
        assert r["kmax_core_mu"] == lm[-1]
    b.close()
