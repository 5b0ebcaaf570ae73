"""The exact counter at the edges of its tiers: vertices whose upper part is
just inside and just outside each bit-matrix size (complete graphs, closed
forms), 4-cycle counters of 32 bits (degrees above 2^16, closed form), cycles
without a top label, and cycles on both sides of the top labels (oracle)."""
from math import comb

import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402


@pytest.mark.parametrize("n", [3, 33, 34, 65, 66, 257, 258, 513, 514, 1025, 1026, 1100])
def test_complete_graphs(n):
    """|U(a)| = n - 1 at the lowest vertex: the last vertex of each tier and
    the first of the next.  Every 4-subset of K_n is a 4-clique."""
    g = gg.complete(n)
    N, C, te = ps.Graph(g.off, g.col).count_exact()
    c4 = comb(n, 4)
    assert C.tolist() == [0, 0, 0, 0, 0, c4]
    assert N.tolist() == [n * comb(n - 1, 3), 12 * c4, 12 * c4, 3 * c4, 6 * c4, c4]
    assert (te.cpu().numpy() == n - 2).all()


@pytest.mark.parametrize("adjacency", [ps.ADJ_SEARCH, ps.ADJ_VTAB])
def test_last_tier_every_adjacency_variant(adjacency):
    g = gg.complete(1030)
    N, C, te = ps.Graph(g.off, g.col, tuning=ps.make_tuning(adjacency=adjacency)).count_exact()
    assert C.tolist() == [0] * 5 + [comb(1030, 4)] and (te.cpu().numpy() == 1028).all()


@pytest.mark.parametrize("hubs, leaves", [(2, 65_535), (2, 65_536), (3, 70_001)])
def test_wide_counters(hubs, leaves):
    """K_{hubs, leaves}: C(hubs, 2) C(leaves, 2) 4-cycles, no triangles; the
    two hubs of a cycle share `leaves` neighbours (16 bits hold 65,535)."""
    h = np.repeat(np.arange(hubs), leaves)
    v = np.tile(np.arange(hubs, hubs + leaves), hubs)
    g = gg.from_pairs(hubs + leaves, np.stack([h, v], axis=1))
    N, C, te = ps.Graph(g.off, g.col).count_exact(max_blocks=4)
    assert int(N[3]) == comb(hubs, 2) * comb(leaves, 2) and N[4] == 0 and N[5] == 0
    assert int(N[0]) == hubs * comb(leaves, 3) + leaves * comb(hubs, 3)
    assert not te.any()


def test_cycles_below_the_top_labels():
    """20,000 disjoint 4-cycles: most have no vertex among the top labels."""
    k = 20_000
    base = 4 * np.arange(k)[:, None] + np.array([[0, 1, 2, 3]])
    pairs = np.concatenate([base[:, [i, (i + 1) % 4]] for i in range(4)])
    N, C, te = ps.Graph(*(lambda g: (g.off, g.col))(gg.from_pairs(4 * k, pairs))).count_exact(max_blocks=3)
    assert N.tolist() == [0, 4 * k, 0, k, 0, 0] and C.tolist() == [0, 0, 0, k, 0, 0]


@pytest.mark.parametrize("n", [16_385, 40_000])
def test_cycles_on_both_sides(n):
    g = gg.chung_lu(n, 9.0, 2.4, 300.0, 5)
    og = O.prepare(g.off, g.col)
    N, C = O.exact_counts(og.off, og.col)
    t = O.triangles_per_edge(og.off, og.col, og.eu, og.ev)
    gN, gC, te = ps.Graph(g.off, g.col).count_exact()
    assert gN.astype(np.int64).tolist() == N.tolist() and gC.tolist() == C.tolist()
    assert np.array_equal(te.cpu().numpy().astype(np.uint32), t)
