"""The radix sort behind the degree order, the edge table and edge-list ingest
at its edges: one tile and its neighbours, the last size whose blocks add up
the digit counts themselves (32 tiles) and the first that scans them, digits
that cross from the larger id's bits into the smaller's, and the smallest ids."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O
from test_gpu_parity import _check_structure

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402


@pytest.mark.parametrize("n, e", [(1, 1), (1, 3), (2, 1), (2, 9), (3, 7), (5, 40), (9, 4095), (300, 4096), (257, 4097),
                                  (4097, 32 * 4096 - 1), (70_000, 32 * 4096), (1 << 17, 32 * 4096 + 1),
                                  ((1 << 18) + 1, 300_001)])
def test_ingest_sizes(n, e):
    """Random pairs with repeats and self-loops: the oracle's CSR."""
    rs = np.random.Generator(np.random.PCG64(n + e))
    src = rs.integers(0, n, e).astype(np.int32)
    dst = np.where(rs.random(e) < 0.05, src, rs.integers(0, n, e)).astype(np.int32)
    if e > 100:
        src[-e // 10:], dst[-e // 10:] = dst[:len(src[-e // 10:])], src[:len(src[-e // 10:])]
    off, col = O.csr_from_edges(n, src, dst)
    g_off, g_col = ps.csr_from_edges(n, src, dst)
    assert np.array_equal(g_off.cpu().numpy(), off) and np.array_equal(g_col.cpu().numpy(), col)


@pytest.mark.parametrize("n", [4095, 4097, 32 * 4096, 32 * 4096 + 1])
def test_structure_at_tile_edges(n):
    """Every load array against the oracle with n vertices and about n (one
    sort tile per sort tile of vertices) to 2 n edges."""
    _check_structure(gg.chung_lu(n, 3.0, 2.5, 60.0, 9, exact_pairs=False))


def test_equal_degrees():
    """All degrees equal: the order is by id alone; and all zero."""
    _check_structure(gg.cycle(5000))
    G = ps.Graph(*(lambda g: (g.off, g.col))(gg.empty(7)))
    assert G.copy(ps.PS_ARRAY_RANK).tolist() == list(range(7)) and G.copy(ps.PS_ARRAY_OFFSETS).tolist() == [0] * 8
