"""Both samplers in one launch (counting a host graph, adaptive runs): the
histograms of the separate samplers, for numbers of samples around the blocks'
and the grid's edges, equal and unequal, none of one kind, and graphs without
centred paths or without paths."""
import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

SEED = 77


def _host(g, k3, kc, tuning=None, spare=0):
    off, col = np.ascontiguousarray(g.off, np.int64), np.ascontiguousarray(g.col, np.int32)
    t = tuning or ps.make_tuning()
    nbytes = ps.ps_end_to_end_workspace_bytes(g.n, col.size, t) + spare
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    base = (ws.data_ptr() + 255) // 256 * 256
    rc, est, lo, hi, h6, h4, st = ps.ps_count_motifs_host(off, col, k3, kc, SEED, 0.01, base, nbytes, t)
    return rc, h6.tolist(), h4.tolist()


def _apart(g, k3, kc, tuning=None):
    G = ps.Graph(g.off, g.col, tuning=tuning)
    h6 = G.sample_3paths(k3, SEED).cpu().numpy().astype(np.uint64)[:6].tolist() if k3 else [0] * 6
    h4 = G.sample_centered(kc, SEED).cpu().numpy().astype(np.uint64)[:4].tolist() if kc else [0] * 4
    return h6, h4


@pytest.mark.parametrize("k3, kc", [(1, 1), (31, 1), (1, 33), (255, 257), (256, 256), (1, 100_003), (100_003, 1), (0, 5000),
                                    (5000, 0), (77_777, 77_823), (155_648, 155_648), (155_649, 1), (300_001, 200_003),
                                    (3_000_017, 999)])
def test_numbers_of_samples(k3, kc):
    g = gg.chung_lu(3000, 10.0, 2.2, 300.0, 8)
    rc, h6, h4 = _host(g, k3, kc)
    assert (h6, h4) == _apart(g, k3, kc)
    assert sum(h6) == k3 and sum(h4) == kc


@pytest.mark.parametrize("adjacency", [0, ps.ADJ_HASH, ps.ADJ_SEARCH, ps.ADJ_VTAB])
@pytest.mark.parametrize("block", [128, 256, 512, 1024])
def test_tunings(adjacency, block):
    g = gg.rmat(10, 8.0, seed=4)
    t = ps.make_tuning(block_size=block, adjacency=adjacency, blocks_per_sm=1 if block > 256 else 0)
    assert _host(g, 50_001, 40_009, t)[1:] == _apart(g, 50_001, 40_009, t)


@pytest.mark.parametrize("order", [0, 1, -1])
def test_scratch_for_the_order(order):
    """Bytes beyond the minimum: drawn in order only where that is asked for."""
    g = gg.chung_lu(3000, 10.0, 2.2, 300.0, 8)
    t = ps.make_tuning(draw_order=order)
    spare = ps.ps_ordered_scratch_bytes(1 << 16)
    assert _host(g, 150_000, 70_001, t, spare)[1:] == _apart(g, 150_000, 70_001)


@pytest.mark.parametrize("name", ["path", "star", "empty", "cycle", "complete"])
def test_small_graphs(name):
    g = {"path": lambda: gg.path(4), "star": lambda: gg.star(9), "empty": lambda: gg.empty(7),
         "cycle": lambda: gg.cycle(5), "complete": lambda: gg.complete(6)}[name]()
    rc, h6, h4 = _host(g, 1000, 1200)
    G = ps.Graph(g.off, g.col)
    a6, a4 = _apart(g, 1000, 1200)
    assert h6 == (a6 if G.stats.W else [0] * 6) and h4 == (a4 if G.stats.Lambda else [0] * 4)
