"""The plain samplers on a graph large enough for fewer resident threads: the
counts are those of any other number of blocks, alone and in one launch."""
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

K, SEED = 1_000_003, 19


@pytest.fixture(scope="module")
def host():
    return gg.rmat(19, 20.0, seed=6)


@pytest.mark.parametrize("adjacency", [ps.ADJ_HASH, ps.ADJ_SEARCH, ps.ADJ_VTAB])
def test_counts_do_not_depend_on_blocks(host, adjacency):
    got = []
    for block, per_sm in ((0, 0), (256, 4), (128, 0), (1024, 0)):
        G = ps.Graph(host.off, host.col, tuning=ps.make_tuning(adjacency=adjacency, block_size=block, blocks_per_sm=per_sm))
        assert int(G.stats.m) >= 1 << 23
        _, h6, h4, *_ = G.count_adaptive(SEED, 1e-9, k0=K, k_max=K)
        got.append([G.sample_3paths(K, SEED).cpu().numpy()[:6].tolist(), G.sample_centered(K, SEED).cpu().numpy()[:4].tolist()])
        assert got[-1] == [h6.tolist(), h4.tolist()]
        G.close()
    assert all(g == got[0] for g in got)
    assert sum(got[0][0]) == K and sum(got[0][1]) == K
