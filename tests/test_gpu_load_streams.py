"""Loads on different streams do not wait for each other: one whose stream is
still busy with earlier work holds up neither the host nor the stream of
another thread's load."""
import threading
import time

import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

BUSY_CYCLES = 3_000_000_000  # 1.5 to 2 s; a load takes well under a millisecond


class _Load:
    def __init__(self, g):
        self.off, self.col = torch.from_numpy(g.off).cuda(), torch.from_numpy(g.col).cuda()
        self.n, self.nnz = g.n, int(g.col.shape[0])
        self.ws = torch.empty(ps.ps_graph_workspace_bytes(self.n, self.nnz), dtype=torch.uint8, device="cuda")
        self.stream = torch.cuda.Stream()

    def run(self):
        self.rc, self.h = ps.ps_load_csr(self.n, self.nnz, self.off.data_ptr(), self.col.data_ptr(),
                                         self.ws.data_ptr(), self.ws.numel(), None, self.stream)

    def columns(self):
        out = np.zeros(self.nnz, dtype=np.int32)
        assert self.rc == ps.PS_OK
        assert ps.ps_graph_copy(self.h, ps.PS_ARRAY_COLUMNS, out.ctypes.data, out.nbytes) == ps.PS_OK
        ps.ps_graph_free(self.h)
        return out


@pytest.mark.parametrize("make", [lambda: gg.chung_lu(3000, 10.0, 2.4, 60.0, 5), lambda: gg.star(6000)],
                         ids=["short rows", "a long row"])
def test_a_load_does_not_wait_for_another_stream(make):
    a, b = _Load(make()), _Load(make())
    torch.cuda.synchronize()

    def both():
        t = threading.Thread(target=b.run)
        t.start()
        time.sleep(0.2)  # b's load is queued and its host thread waits
        a.run()
        return t

    both().join()  # kernels and streams in place
    want = a.columns()
    assert b.columns().tolist() == want.tolist()
    # streams that share one of the device's few hardware queues do wait for
    # each other, so one of a few pairs of streams has to pass
    waited = []
    while len(waited) < 4 and all(waited):
        a.stream, b.stream = torch.cuda.Stream(), torch.cuda.Stream()
        with torch.cuda.stream(b.stream):
            torch.cuda._sleep(BUSY_CYCLES)
            done = torch.cuda.Event()
            done.record(b.stream)
        t = both()
        waited.append(done.query())
        t.join()
        assert a.columns().tolist() == want.tolist() and b.columns().tolist() == want.tolist()
    assert not all(waited)


def test_more_loads_than_side_streams():
    loads = [_Load(gg.chung_lu(2000 + i, 8.0, 2.3, 300.0, i)) for i in range(24)]
    torch.cuda.synchronize()
    for load in loads:
        load.run()
    want = [load.columns().tolist() for load in loads]
    threads = []
    for load in loads:  # each waits on the host with its streams taken
        with torch.cuda.stream(load.stream):
            torch.cuda._sleep(BUSY_CYCLES // 10)
        threads.append(threading.Thread(target=load.run))
        threads[-1].start()
    for t in threads:
        t.join()
    assert [load.columns().tolist() for load in loads] == want
