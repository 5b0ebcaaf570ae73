"""Rows of at most 32 entries, several to a warp where there are more rows than
warps: lengths around 8, 16 and 32, numbers of rows that leave a group short,
and a repeated entry, a self-loop and a bad column in such rows."""
from types import SimpleNamespace

import numpy as np
import pytest

import graphgen as gg
import oracle as O
from test_gpu_parity import _check_structure

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1411_4942_gb300 import pathsample as ps  # noqa: E402


def _blocks(*sizes):
    """Disjoint complete graphs: rows of exactly size - 1 entries."""
    src, dst, at = [], [], 0
    for s in sizes:
        i, j = np.triu_indices(s, 1)
        src.append(at + i)
        dst.append(at + j)
        at += s
    return O.csr_from_edges(at, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32))


@pytest.mark.parametrize("sizes", [(9,) * 3001, (10,) * 2500 + (17,) * 400 + (18,) * 301,
                                   (33,) * 700 + (34,) * 5 + (2,) * 9000, tuple(range(2, 40)) * 40])
def test_exact_lengths(sizes):
    off, col = _blocks(*sizes)
    _check_structure(SimpleNamespace(off=off, col=col), ps.Graph(off, col))


@pytest.mark.parametrize("n, mean", [(19_500, 5.0), (40_001, 9.0), (60_002, 14.0), (30_003, 25.0)])
def test_mixed_lengths(n, mean):
    _check_structure(gg.chung_lu(n, mean, 2.5, 300.0, 5, exact_pairs=False))


@pytest.mark.parametrize("n", [50, 30_000])
@pytest.mark.parametrize("what", ["repeat", "loop", "column"])
def test_bad_rows(n, what):
    g = gg.cycle(n)
    off, col = np.array(g.off), np.array(g.col)
    at = int(off[n // 2])
    if what == "repeat":
        col[at] = col[at + 1]
    elif what == "loop":
        col[at] = n // 2
    else:
        col[at] = n
    want = O.validate(off, col)
    assert want == (O.ERR_ARG if what == "column" else O.ERR_NOT_SIMPLE)
    with pytest.raises(ps.PathSampleError) as e:
        ps.Graph(off, col)
    assert e.value.code == want
