"""Repeated neighbours in a row sorted through the bitmap: the load reports
them, and every column it has written by then is a label (the kernels that run
before the verdict index by them), whatever the workspace held before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

N, DEG = 6000, 5000  # vertex 0 joined to 1 .. DEG: a row above 4096 entries


def _star():
    off = np.zeros(N + 1, dtype=np.int64)
    off[1:DEG + 2] = DEG + np.arange(DEG + 1)
    off[DEG + 2:] = 2 * DEG
    col = np.zeros(2 * DEG, dtype=np.int32)
    col[:DEG] = np.arange(1, DEG + 1)
    return off, col


def _load(off, col, ws):
    d_off, d_col = torch.from_numpy(off).cuda(), torch.from_numpy(col).cuda()
    return ps.ps_load_csr(N, col.shape[0], d_off.data_ptr(), d_col.data_ptr(), ws.data_ptr(), ws.numel())


@pytest.mark.parametrize("distinct", [1, 2, DEG // 2, DEG - 1])
def test_columns_stay_labels(distinct):
    off, col = _star()
    ws = torch.full((ps.ps_graph_workspace_bytes(N, col.shape[0]),), 0x7F, dtype=torch.uint8, device="cuda")
    rc, h = _load(off, col, ws)
    assert rc == ps.PS_OK
    good = np.zeros(col.shape[0], dtype=np.int32)
    assert ps.ps_graph_copy(h, ps.PS_ARRAY_COLUMNS, good.ctypes.data, good.nbytes) == ps.PS_OK
    ps.ps_graph_free(h)
    host = ws.cpu().numpy()
    at = [a for a in range(0, host.size - good.nbytes + 1, 256) if host[a:a + good.nbytes].tobytes() == good.tobytes()]
    assert len(at) == 1  # where the workspace holds the columns
    col[:DEG] = 1 + np.arange(DEG) % distinct
    ws.fill_(0x7F)
    rc, h = _load(off, col, ws)
    assert rc == ps.PS_ERR_NOT_SIMPLE and h is None
    torch.cuda.synchronize()
    got = ws[at[0]:at[0] + good.nbytes].view(torch.int32)
    assert int(got.min()) >= 0 and int(got.max()) < N
