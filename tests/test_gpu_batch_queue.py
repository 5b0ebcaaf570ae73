"""The batched launch's queue at its edges: fewer items than blocks, the last
number of items that is claimed one at a time and the first that is claimed
ahead, many more than that; items that change graph every time, name no graph,
or name a graph of another adjacency variant; an item list that is only 8-byte
aligned."""
import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import batch as psb  # noqa: E402
from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

SEED = 31


@pytest.fixture(scope="module")
def graphs():
    hosts = [gg.chung_lu(3000, 10.0, 2.2, 300.0, 8), gg.rmat(11, 8.0, seed=4), gg.complete(30)]
    return [ps.Graph(g.off, g.col) for g in hosts]


def _launch(gset, items, slots, skew=0):
    """Runs the items (one block per SM, so the queue's length in blocks is
    known) and returns (slot histograms, skipped items)."""
    raw = torch.zeros(items.nbytes + 16, dtype=torch.uint8, device="cuda")
    raw[skew:skew + items.nbytes] = torch.from_numpy(items.view(np.uint8).copy()).cuda()
    hist = torch.zeros(6 * slots, dtype=torch.int64, device="cuda")
    counter = torch.zeros(2, dtype=torch.int32, device="cuda")
    rc = ps.ps_batch_sample_prepared(gset.table.data_ptr(), len(gset), raw.data_ptr() + skew, items.shape[0],
                                     hist.data_ptr(), counter.data_ptr(), ps.make_tuning(block_size=128, blocks_per_sm=1))
    assert rc == ps.PS_OK
    return hist.cpu().numpy().reshape(slots, 6), int(counter[1])


def _plain(G, sampler, k):
    h = (G.sample_3paths if sampler == 0 else G.sample_centered)(k, SEED).cpu().numpy()[:6]
    return (h if sampler == 0 else np.concatenate([h[:4], [0, 0]])).tolist()


@pytest.mark.parametrize("skew", [0, 8])
@pytest.mark.parametrize("per_block", [0, 4, 4.01, 9.5])
def test_queue_lengths(graphs, per_block, skew):
    blocks = torch.cuda.get_device_properties(0).multi_processor_count
    n = max(1, int(round(per_block * blocks)))
    gset = psb.GraphSet(graphs)
    # item i: ids [37 q, 37 (q + 1)) of graph i % 3, sampler (i / 3) % 2
    items = np.zeros(n, dtype=ps.WORK_DTYPE)
    i = np.arange(n)
    items["graph"], items["sampler"] = i % 3, (i // 3) % 2
    items["slot"] = 2 * items["graph"] + items["sampler"]
    items["first_id"], items["count"], items["seed"] = 37 * (i // 6), 37, SEED
    hist, skipped = _launch(gset, items, 6, skew)
    assert skipped == 0
    for s in range(6):
        k = 37 * int((items["slot"] == s).sum())
        assert hist[s].tolist() == (_plain(graphs[s // 2], s % 2, k) if k else [0] * 6)


@pytest.mark.parametrize("n", [5, 4000])
def test_items_that_do_not_run(graphs, n):
    """Every third item names no graph (not counted, nothing sampled); with a
    graph of another variant in the table the mixed kernel runs every item."""
    other = ps.Graph(*(lambda g: (g.off, g.col))(gg.complete(12)), tuning=ps.make_tuning(adjacency=ps.ADJ_SEARCH))
    gset = psb.GraphSet([graphs[0], other])
    items = np.zeros(n, dtype=ps.WORK_DTYPE)
    i = np.arange(n)
    items["graph"] = np.where(i % 3 == 2, 99, i % 3)
    items["slot"] = np.where(i % 3 == 2, 2, i % 3)
    items["first_id"], items["count"], items["seed"] = 11 * (i // 3), 11, SEED
    hist, skipped = _launch(gset, items, 3)
    assert skipped == 0 and not hist[2].any()
    for s, G in enumerate((graphs[0], other)):
        assert hist[s].tolist() == _plain(G, 0, 11 * int((i % 3 == s).sum()))


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("name", [99, 0xFFFFFFFE, 0xFFFFFFFF])
@pytest.mark.parametrize("n", [1, 3000])
def test_blocks_that_start_on_an_item_without_a_graph(graphs, n, name, mixed):
    """The queue opens with items that name no graph, so that every block's
    first one is such an item: nothing sampled, none counted as skipped, and
    the items behind them run."""
    second = graphs[1]
    if mixed:
        g = gg.complete(12)
        second = ps.Graph(g.off, g.col, tuning=ps.make_tuning(adjacency=ps.ADJ_SEARCH))
    gset = psb.GraphSet([graphs[0], second])
    items = np.zeros(n + 6, dtype=ps.WORK_DTYPE)
    items["graph"][:n], items["slot"][:n] = name, 2
    i = np.arange(6)
    items["graph"][n:] = items["slot"][n:] = i % 2
    items["first_id"][n:] = 11 * (i // 2)
    items["sampler"][:n] = np.arange(n) % 2
    items["count"], items["seed"] = 11, SEED
    hist, skipped = _launch(gset, items, 3)
    assert skipped == 0 and not hist[2].any()
    for s, G in enumerate((graphs[0], second)):
        assert hist[s].tolist() == _plain(G, 0, 33)
