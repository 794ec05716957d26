"""The gathers over the interleaved columns of the short lists, at the edges of
the degree bins: groups of one to a few slices on either side of each bin."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


def binned(count):
    """count vertices of each degree at the bins' edges, on 1030 shared leaves."""
    e, n = [], 1030
    for d in (1, 2, 4, 5, 31, 32, 33, 64, 255, 256, 257, 1023, 1024, 1025):
        for i in range(count):
            e += [(n, (7 * i + k) % 1030) for k in range(d)]
            n += 1
    return inputs.from_edges(n, e)


@pytest.mark.parametrize("count", [1, 31, 32, 33])
@pytest.mark.parametrize("light", [4, 32, 256])
def test_gathers_at_bin_edges(count, light):
    off, col = binned(count)
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        g.set_pull_light(light)
        c.set_option(lgc.OPT_PULL, 2)
        c.set_option(lgc.OPT_SWEEP_CROSS, 2)
        ref = oracle.hkpr(off, col, 5, 5.0, 8, 1e-7)
        for mode in ("det", "atomic"):
            p, st = lgc.hkpr(g, 5, 5.0, 8, 1e-7, mode=mode)
            assert st.pushed_edges == ref.pushed_edges
            assert np.array_equal(p.idx, ref.idx)
            if mode == "det":
                assert np.array_equal(p.val, ref.val)
            else:  # eight rounds, each within two roundings of the fold of 1025 or fewer
                assert np.abs(p.val - ref.val).sum() <= 8 * 1025 * 2.0 ** -53 * ref.val.sum()
        # supports above and below a quarter of the vertices
        for eps in (1e-7, 3e-5, 3e-4):
            p, st = lgc.prnibble(g, 5, 0.05, eps, mode="det")
            ref = oracle.prnibble(off, col, 5, 0.05, eps)
            assert np.array_equal(p.idx, ref.idx) and np.array_equal(p.val, ref.val)
            rs = oracle.sweep(off, col, ref.idx, ref.val)
            s = lgc.sweep(g, p)
            assert (s.size, s.vol, s.cut) == (rs.best, rs.best_vol, rs.best_cut)
            assert np.array_equal(s.ids, rs.cluster)
    finally:
        g.close()
        c.close()
