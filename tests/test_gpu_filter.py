"""The default adjacency test (hub rows, edge filter, sorted rows) against the
oracle where it can go wrong: no hub rows at all (every pair asks the filter),
a few hub rows over a narrow span, dense graphs (most filter hits are edges)
and graphs small enough for the smallest filter."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import batch as psb  # noqa: E402
from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

GRAPHS = {
    "P5": lambda: gg.path(5),
    "K40": lambda: gg.complete(40),
    "gnp150": lambda: gg.gnp(150, 0.5, 3),
    "rmat12": lambda: gg.rmat(12, 8.0, seed=4),
    "cl20000": lambda: gg.chung_lu(20000, 15.0, 2.1, 1500.0, 12),
}
HUBS = {"none": dict(hub_count=-1), "narrow": dict(hub_count=31, hub_span_log2=5, hub_min_degree=1),
        "wide": dict(hub_count=40, hub_span_log2=-1, hub_min_degree=1)}


@pytest.mark.parametrize("hubs", list(HUBS))
@pytest.mark.parametrize("name", list(GRAPHS))
def test_filter_answers_equal_oracle(name, hubs):
    g = GRAPHS[name]()
    og = O.prepare(g.off, g.col)
    k, seed, first = 40_009, 77, 2 ** 33 - 5
    want6 = O.sample_3paths(og, k, seed, first, threads=8).tolist() if og.W else [0] * 6
    want4 = O.sample_centered(og, k, seed, first, threads=8).tolist() if og.Lambda else [0] * 4
    G = ps.Graph(g.off, g.col, tuning=ps.make_tuning(draw_order=1, **HUBS[hubs]))
    got = [(G.sample_3paths(k, seed, first), G.sample_centered(k, seed, first)),
           (G.sample_3paths_ordered(k, seed, first), G.sample_centered_ordered(k, seed, first))]
    for h6, h4 in got:
        assert h6.cpu().numpy()[:6].tolist() == want6 and h4.cpu().numpy()[:4].tolist() == want4
    for spt in (1, 2):
        runner = psb.BatchRunner(psb.GraphSet([G]), [psb.Request(0, 0, k, seed, first), psb.Request(0, 1, k, seed, first)],
                                 psb.LaunchConfig(block_size=128, chunk=1 << 12, samples_per_thread=spt))
        runner.launch()
        h = runner.histograms().astype(np.int64)
        assert h[0].tolist() == want6 and h[1].tolist() == want4 + [0, 0]
