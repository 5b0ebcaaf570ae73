"""Filter hits confirmed in the sorted rows: graphs in which nearly every pair
asked is an edge, without hub rows, with rows around the lengths at which the
search takes another step (9 to 10, 36 to 43, 150) and column arrays that end
inside a 16-byte block.  Counts equal the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import batch as psb  # noqa: E402
from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

SEED, K = 77, 6000


def _ring(n, d):
    """Every vertex joined to its d / 2 nearest on either side."""
    return gg.from_pairs(n, [(v, (v + s) % n) for v in range(n) for s in range(1, d // 2 + 1)])


GRAPHS = {**{f"complete {n}": (lambda n=n: gg.complete(n)) for n in (4, 5, 9, 10, 11, 12, 14, 36, 37, 38, 39, 42, 44, 151)},
          **{f"ring {d}": (lambda d=d: _ring(301, d)) for d in (4, 8, 10, 12, 36, 38, 60)},
          "cliques of two sizes": lambda: gg.from_pairs(90, [(a, b) for lo, hi in ((0, 45), (30, 90)) for a in range(lo, hi)
                                                            for b in range(a + 1, hi) if (a * b) % 7])}


@pytest.mark.parametrize("name", GRAPHS)
def test_hits_confirmed(name):
    g = GRAPHS[name]()
    og = O.prepare(g.off, g.col)
    G = ps.Graph(g.off, g.col, tuning=ps.make_tuning(hub_count=-1))
    want = [np.asarray(O.sample_3paths(og, K, SEED)).tolist(), np.asarray(O.sample_centered(og, K, SEED)).tolist()]
    got = [G.sample_3paths(K, SEED).cpu().numpy()[:6].tolist(), G.sample_centered(K, SEED).cpu().numpy()[:4].tolist()]
    assert got == want
    gset = psb.GraphSet([G])
    for spt in (1, 2):
        run = psb.BatchRunner(gset, [psb.Request(0, s, K, SEED) for s in (0, 1)], psb.LaunchConfig(128, 500, 0, spt))
        run.launch()
        h = run.histograms().tolist()
        assert [h[0], h[1][:4]] == want
