"""HK-PR levels whose threshold is zero: (e^t eps) / (2 N psi_j) underflows at
a subnormal eps, or at a large t with the exponent's other sign."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu

CASES = {"subnormal": (5.0, 12, 5e-324, 1), "not_zero": (3.0, 9, 1.5e-322, 1),
         "other_sign": (400.0, 450, 1e-7, -1)}


@pytest.mark.parametrize("device", [1, 0])
@pytest.mark.parametrize("mode", ["det", "atomic"])
@pytest.mark.parametrize("case", list(CASES))
def test_zero_thresholds(case, mode, device):
    """Such a level's frontier is every vertex its set holds."""
    t, N, eps, sign = CASES[case]
    off, col = inputs.random_graph(60, 150, seed=2)
    x = int(np.flatnonzero(np.diff(off) >= 1)[0])
    ref = oracle.hkpr(off, col, x, t, N, eps, threshold_sign=sign)
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        c.set_option(lgc.OPT_DEVICE_ROUNDS, device)
        c.set_option(lgc.OPT_HK_THRESHOLD_SIGN, sign)
        p, st = lgc.hkpr(g, x, t, N, eps, mode=mode)
        assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes,
                                                           ref.pushed_edges)
        assert np.array_equal(p.idx, ref.idx)
        if mode == "det":
            assert np.array_equal(p.val, ref.val)
        else:  # the order of the adds of at most N rounds, each of at most 59 terms
            assert np.abs(p.val - ref.val).sum() <= N * 59 * 2.0 ** -53 * ref.val.sum()
    finally:
        g.close()
        c.close()
