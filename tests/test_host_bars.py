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


@pytest.mark.parametrize("k, c, delta", [
    (20601542668580, 20601542668542, 6.501372376723512e-92),
    (105277841728479, 105277841728475, 0.004123769651538563),
    (6968, 6942, 1e-305), (89765, 89760, 2.3e-50), (154357, 154326, 1e-317), (121166605, 121166564, 1e-308),
    (1498341142809319936, 1466, 3e-308), (1568932294595252992, 1452, 1e-308),
] + [(k, k - r, 10.0 ** -e) for k in (1000, 24001, 10 ** 6 + 3, (1 << 30) + 1, 1 << 45)
     for r in (1, 4, 15, 40) for e in (2, 30, 90, 150, 200, 250, 300)])
def test_bars_next_to_the_ends(k, c, delta):
    """Roots within a few ulp of 1 or of alpha, where D is steep or flat and
    Newton's last step says little about how far the root is."""
    st = ps.PsStats()
    st.W, st.Lambda, st.N1_lo, st.n, st.m = 1 << 40, 1 << 38, 10 ** 7, 10, 9
    h6 = np.array([0, c, k - c, c, c, k - c], dtype=np.uint64)
    h4 = np.array([0, c, k - c, c], dtype=np.uint64)
    rc, est, lo, hi = ps.ps_estimate(st, h6, k, h4, k, delta)
    _, oest, olo, ohi = O.estimate(int(st.W), int(st.Lambda), st.N1, h6, k, h4, k, delta)
    assert est.tolist() == list(oest) and lo.tolist() == list(olo) and hi.tolist() == list(ohi)
