"""Minimum cuts whose rounds mix nodes taken by warps (at most 2,048 arcs) and
nodes taken by blocks (more): both kinds run in one launch and push into one
another.  Answers are compared with the oracle's Algorithm 1 exactly.
"""
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


def _graph(kind):
    if kind == "clique64":      # h = 3: 2,018 arcs a vertex, all small
        return gg.random_small(64, 1.0, seed=1)
    if kind == "clique65":      # 2,082 arcs, all big
        return gg.random_small(65, 1.0, seed=1)
    if kind == "mixed":         # about 2,075 arcs a vertex, on both sides of the line
        return gg.random_small(90, 0.8, seed=2)
    if kind == "lopsided":      # a dense part inside a thinner one
        n, s, d = gg.random_small(110, 0.25, seed=3)
        n, s, d, _ = gg.plant(n, s, d, 75, 0.9, 4)
        return n, s, d
    # h = 2: five hubs of 2,100 neighbours each, adjacent to one another
    hubs, leaves = 5, 2100
    a = np.repeat(np.arange(hubs, dtype=np.uint32), leaves)
    b = np.tile(np.arange(hubs, hubs + leaves, dtype=np.uint32), hubs)
    i, j = np.triu_indices(hubs, 1)
    rng = np.random.default_rng(5)
    x, y = (rng.integers(hubs, hubs + leaves, 3000, dtype=np.uint32) for _ in range(2))
    return (hubs + leaves, np.concatenate([a, i.astype(np.uint32), x]),
            np.concatenate([b, j.astype(np.uint32), y]))


@pytest.mark.parametrize("kind,h", [("clique64", 3), ("clique65", 3), ("mixed", 3),
                                    ("lopsided", 3), ("hubs", 2)])
def test_exact_mixed_rounds(L, orc, kind, h):
    n, s, d = _graph(kind)
    w = orc.exact_cds(orc.csr(n, s, d), h)
    with L.Graph.from_edges(n, s, d) as g:
        for _ in range(2):      # the second cut starts from used buffers
            r = g.core_exact(h)
            assert (r["mu"], r["size"]) == (w["mu"], w["size"])
            assert np.array_equal(np.asarray(r["cds"], np.uint32), w["cds"])
