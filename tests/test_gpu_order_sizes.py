"""The draw order at the sizes where its plan changes: one bucket and two, a
bucket just full and one id more, both tile lengths, more ids than are sorted
at once; with a scratch of exactly the documented size, whose surroundings must
stay untouched."""
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

GUARD = 4096


@pytest.fixture(scope="module")
def graph():
    g = gg.chung_lu(3000, 12.0, 2.3, 200.0, 2)
    return ps.Graph(g.off, g.col, tuning=ps.make_tuning(draw_order=1))


@pytest.mark.parametrize("k, chunk", [(1, 1), (31, 31), (8191, 8191), (8192, 8192), (8193, 8193), (16385, 16385),
                                      (32768, 32768), (32769, 32769), (65537, 65537),
                                      (100_003, 100_003), ((1 << 22) - 1, (1 << 22) - 1), (1 << 22, 1 << 22),
                                      ((1 << 22) + 1, (1 << 22) + 1), (10_000_019, 10_000_019), (50_000, 8193),
                                      (100_000, 32769),
                                      ((1 << 26) + 77, (1 << 26) + 77), ((1 << 27) + 5, (1 << 27) + 5)])
def test_plan_edges(graph, k, chunk):
    nbytes = ps.ps_ordered_scratch_bytes(chunk)
    buf = torch.full((nbytes + 2 * GUARD,), 0x5A, dtype=torch.uint8, device="cuda")
    seed, first = 91, 2 ** 32 - 1000
    for plain, ordered in ((graph.sample_3paths, ps.ps_sample_3paths_ordered),
                           (graph.sample_centered, ps.ps_sample_centered_ordered)):
        hist = graph.new_hist()
        rc = ordered(graph.handle, k, seed, first, hist.data_ptr(), buf.data_ptr() + GUARD, nbytes)
        assert rc == ps.PS_OK
        assert hist.tolist() == plain(k, seed, first).tolist()
    assert (buf[:GUARD] == 0x5A).all() and (buf[GUARD + nbytes:] == 0x5A).all()
