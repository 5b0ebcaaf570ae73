"""The error bars' root search (Newton, then only the halvings near the root
evaluated) against the oracle's plain bisection, bit for bit, where the roots
are hardest: counts of 1 and k - 1, few and very many samples, loose and very
tight confidences."""
import numpy as np
import pytest

import oracle as O
from paper_1411_4942_gb300 import pathsample as ps


@pytest.mark.parametrize("delta", [0.9, 0.5, 0.01, 1e-6, 1e-12])
@pytest.mark.parametrize("k", [2, 3, 12, 1958, 3_437_001, 1 << 27, (1 << 40) + 7])
def test_bars_equal_plain_bisection(k, delta):
    st = ps.PsStats()
    st.W, st.Lambda, st.N1_lo, st.n, st.m = 10 ** 9 + 7, 10 ** 8 + 3, 10 ** 7, 10, 9
    for c in sorted({1, 2, k // 1000 + 1, k // 3 + 1, k // 2, k - 1}):
        if not 0 < c < k:
            continue
        h6 = np.array([0, c, k - c, c, 1, c], dtype=np.uint64)
        h4 = np.array([0, c, k - c, 1], dtype=np.uint64)
        rc, est, lo, hi = ps.ps_estimate(st, h6, k, h4, k, delta)
        _, oest, olo, ohi = O.estimate(int(st.W), int(st.Lambda), st.N1, h6, k, h4, k, delta)
        assert est.tolist() == list(oest) and lo.tolist() == list(olo) and hi.tolist() == list(ohi)
