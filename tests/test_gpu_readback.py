"""Small results read back through pinned slots: more threads at once than
there are slots (the rest copy), each on a stream of its own, must all see
their own results."""
import threading

import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

THREADS = 48


def test_more_threads_than_slots():
    g = gg.chung_lu(2000, 10.0, 2.2, 200.0, 3)
    graph = ps.Graph(g.off, g.col)
    want = [graph.count_adaptive(seed, 0.02, k0=1 << 12, k_max=1 << 15) for seed in range(THREADS)]
    got = [None] * THREADS
    gate = threading.Barrier(THREADS)

    def work(seed):
        with torch.cuda.stream(torch.cuda.Stream()):
            gate.wait()
            for _ in range(3):
                got[seed] = graph.count_adaptive(seed, 0.02, k0=1 << 12, k_max=1 << 15)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(THREADS)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(want, got):
        assert b is not None and a[0] == b[0]
        assert all(np.array_equal(np.asarray(x), np.asarray(y)) for x, y in zip(a[1:], b[1:]))
