"""The radix sort behind the degree order, the edge table and edge-list ingest
at its edges: one tile and its neighbours, the last size whose blocks add up
the digit counts themselves (64 tiles) and the first that scans them, digits
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
                                  (300, 3583), (300, 3584), (300, 3585), (4097, 64 * 3584), (4097, 64 * 3584 + 1),
                                  (4097, 64 * 4096 - 1), (70_000, 64 * 4096), (1 << 17, 64 * 4096 + 1),
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


@pytest.mark.parametrize("n", [255, 257, 4095, 4097, 65_535, 65_537, 64 * 3584, 64 * 3584 + 1, 64 * 4096,
                               64 * 4096 + 1])
def test_structure_at_tile_edges(n):
    """Every load array against the oracle with n vertices and about n (one
    sort tile per sort tile of vertices) to 2 n edges."""
    _check_structure(gg.chung_lu(n, 3.0, 2.5, 60.0, 9, exact_pairs=False))


@pytest.mark.parametrize("n", [3, 200, 256, 5000, 1 << 20])
@pytest.mark.parametrize("e", [31, 1023, 1024, 1025, 2049, 4097, 8192, 8193, 16_385, 40_000, 65_536, 131_071,
                               131_072, 131_073])
def test_one_cluster(n, e):
    """The sort of short lists in one launch: one block and the first of two,
    four, eight and sixteen, rows just full and one item more, the largest list and the
    first that is sorted pass by pass; with repeats, so the second sort is
    shorter than its launch."""
    rs = np.random.Generator(np.random.PCG64(n + e))
    src, dst = rs.integers(0, n, e).astype(np.int32), rs.integers(0, n, e).astype(np.int32)
    off, col = O.csr_from_edges(n, src, dst)
    g_off, g_col = ps.csr_from_edges(n, src, dst)
    assert np.array_equal(g_off.cpu().numpy(), off) and np.array_equal(g_col.cpu().numpy(), col)


@pytest.mark.parametrize("n", [1024, 1025, 8193, 16_385, 65_536, 100_003, 131_072, 131_073])
def test_one_cluster_structure(n):
    """Degree order and edge table from lists sorted in one launch."""
    _check_structure(gg.chung_lu(n, 2.0, 2.5, 40.0, 9, exact_pairs=False))


def test_equal_degrees():
    """All degrees equal: the order is by id alone; and all zero."""
    _check_structure(gg.cycle(5000))
    G = ps.Graph(*(lambda g: (g.off, g.col))(gg.empty(7)))
    assert G.copy(ps.PS_ARRAY_RANK).tolist() == list(range(7)) and G.copy(ps.PS_ARRAY_OFFSETS).tolist() == [0] * 8


@pytest.mark.parametrize("bad_column", [False, True])
@pytest.mark.parametrize("n", [3, 300, 70_000])
def test_rows_too_long(n, bad_column):
    """A row of more than n - 1 entries ends the load before its rows are
    walked; a column out of range outranks it, as for the oracle."""
    d = n + 5
    off = np.concatenate([[0], np.full(n, d)]).astype(np.int64)
    col = (1 + np.arange(d) % max(n - 1, 1)).astype(np.int32)
    if bad_column:
        col[-1] = n
    want = O.validate(off, col)
    assert want == (O.ERR_ARG if bad_column else O.ERR_NOT_SIMPLE)
    t_off, t_col = torch.as_tensor(off, device="cuda"), torch.as_tensor(col, device="cuda")
    nb = ps.ps_graph_workspace_bytes(n, d)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    rc, h = ps.ps_load_csr(n, d, t_off.data_ptr(), t_col.data_ptr(), ws.data_ptr(), nb)
    assert rc == want and h is None
