"""Sorts by counting: supports around the largest size of the 64-bit keys
(20480), with many equal keys, at sizes off the tiles."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0", [1025, 1039, 4095, 16385, 20479, 20480, 20481, 24001])
@pytest.mark.parametrize("ties", [False, True])
def test_sweep_order(n0, ties):
    off, col = inputs.rmat(16, seed=1)
    d = np.diff(off)
    rng = np.random.default_rng(n0)
    idx = np.sort(rng.choice(np.flatnonzero(d > 0), size=n0, replace=False)).astype(np.int32)
    # p/d among 16 values, or all different
    val = d[idx] * 2.0 ** -rng.integers(1, 17, n0) if ties else rng.random(n0) ** 2
    val[rng.random(n0) < 0.01] = 0.0
    ref = oracle.sweep(off, col, idx, val)
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        s = lgc.sweep(g, lgc.host_svec(idx, val))
        assert (s.size, s.vol, s.cut) == (ref.best, ref.best_vol, ref.best_cut)
        assert np.array_equal(s.ids, ref.cluster) and s.conductance == ref.conductance
    finally:
        g.close()
        c.close()
