"""Rows above 4096 entries on a graph of more than 2^20 vertices: lengths just
above the limit, around multiples of the block's slices and far above, with
labels over all 21 bits; and a repeated entry in such a row."""
from types import SimpleNamespace

import numpy as np
import pytest

import oracle as O
from test_gpu_parity import _check_structure

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402

N = (1 << 20) + 12_345


def _hubs(lengths, seed):
    rs = np.random.Generator(np.random.PCG64(seed))
    src, dst = [], []
    for i, d in enumerate(lengths):
        ends = rs.choice(N - len(lengths), d, replace=False) + len(lengths)
        src.append(np.full(d, i))
        dst.append(ends)
    # some edges among the rest, so that labels spread over degrees
    a, b = rs.integers(len(lengths), N, (2, 50_000))
    src.append(a[a != b])
    dst.append(b[a != b])
    return O.csr_from_edges(N, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32))


@pytest.mark.parametrize("lengths", [(4097,), (4097, 4128, 4129, 5000), (8191, 8192, 8193, 65_537), (100_001, 4100, 33_333)])
def test_lengths(lengths):
    off, col = _hubs(lengths, sum(lengths))
    _check_structure(SimpleNamespace(off=off, col=col), ps.Graph(off, col))


def test_repeat():
    off, col = _hubs((6000, 9001), 3)
    col = np.array(col)
    col[off[1] + 17] = col[off[1] + 4000]
    assert O.validate(off, col) == O.ERR_NOT_SIMPLE
    with pytest.raises(ps.PathSampleError) as e:
        ps.Graph(off, col)
    assert e.value.code == O.ERR_NOT_SIMPLE
