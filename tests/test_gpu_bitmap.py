"""The block-level bitmap search at the sizes where its layout changes: word
and stride boundaries, node sets above the list buffer, 32- and 64-bit
counters.  Closed forms on K_n and the oracle on random graphs."""
from __future__ import annotations

import math

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


@pytest.mark.parametrize("n,hs", [(34, (4, 5, 8)), (66, (4, 5, 6)), (130, (4, 5, 6)),
                                  (258, (4, 5)), (300, (4, 5)), (1024, (4,)), (1025, (4,))])
def test_complete_graphs(L, n, hs):
    s, d = np.triu_indices(n, 1)
    with L.Graph.from_edges(n, s.astype(np.uint32), d.astype(np.uint32)) as g:
        for h in hs:
            deg, mu = g.clique_degrees(h)
            assert mu == math.comb(n, h)
            assert np.all(deg == math.comb(n - 1, h - 1))


@pytest.mark.parametrize("n,p,h", [(97, 0.6, 7), (200, 0.5, 6), (330, 0.4, 5), (520, 0.3, 4),
                                   (700, 0.15, 4)])
def test_random_dense(L, orc, n, p, h):
    n, s, d = gg.er(n, p, seed=n + h)
    og = orc.csr(n, s, d)
    wdeg, wmu = orc.clique_degrees(og, h)
    with L.Graph.from_edges(n, s, d) as g:
        deg, mu = g.clique_degrees(h)
        core, k = g.core_decompose(h) if n <= 330 and h <= 5 else (None, None)
    assert mu == wmu and np.array_equal(deg, wdeg)
    if core is not None:
        wcore, wk = orc.core_decompose(og, h)
        assert k == wk and np.array_equal(core, wcore)


@pytest.mark.parametrize("n,p,h", [(36, 0.97, 5), (70, 0.95, 5), (105, 0.9, 5), (136, 0.97, 5),
                                   (150, 0.85, 5), (80, 0.9, 6), (60, 0.9, 7)])
def test_register_search(L, orc, n, p, h):
    """Sets of up to and just above 32, 64, 96 and 128 members below a node."""
    n, s, d = gg.er(n, p, seed=3 * n + h)
    wdeg, wmu = orc.clique_degrees(orc.csr(n, s, d), h)
    with L.Graph.from_edges(n, s, d) as g:
        deg, mu = g.clique_degrees(h)
    assert mu == wmu and np.array_equal(deg, wdeg)


@pytest.mark.parametrize("d", [31, 32, 33, 63, 64, 1024, 1025, 12288, 12289])
def test_noalloc_row_tiers(L, d):
    """dsd_triangle_degrees_noalloc on both sides of its row tiers: a hub of
    exactly d higher-id neighbours, which carry edges of their own."""
    import torch
    rng = np.random.default_rng(d)
    n = d + 40
    ring = np.arange(1, d + 1)
    a = rng.integers(1, n, 6 * n)
    b = rng.integers(1, n, 6 * n)
    near = np.minimum(ring + rng.integers(1, 9, d), n - 1)
    s = np.concatenate([np.zeros(d, np.int64), ring, a]).astype(np.uint32)
    t = np.concatenate([ring, near, b]).astype(np.uint32)
    with L.Graph.from_edges(n, s, t) as g:
        want, wmu = g.clique_degrees(3)
        off, adj = g.csr(mem="device")
    deg = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    mu = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    L.dsd_triangle_degrees_noalloc(n, off.data_ptr(), adj.data_ptr(), deg.data_ptr(),
                                   mu.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert int(mu.item()) == wmu
    assert np.array_equal(deg.cpu().numpy().astype(np.uint64), want)
