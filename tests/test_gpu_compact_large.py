"""Dense filters and extraction over more than 2^24 vertices, where the tiles'
counts are added up in groups."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import lgc

pytestmark = pytest.mark.gpu


def spread_star(n, step):
    """Vertex 3 joined to every step-th vertex."""
    leaf = np.arange(0, n, step, dtype=np.int32)
    leaf = leaf[leaf != 3]
    deg = np.zeros(n, np.int64)
    deg[leaf] = 1
    deg[3] = len(leaf)
    off = np.zeros(n + 1, np.int64)
    np.cumsum(deg, out=off[1:])
    col = np.full(int(off[-1]), 3, np.int32)
    col[off[3]:off[4]] = leaf
    return off, col


@pytest.mark.parametrize("n", [(1 << 24) + 2048, 37_000_007])
def test_spread_star(n):
    off, col = spread_star(n, 16)
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        c.set_option(lgc.OPT_DEVICE_ROUNDS, 0)
        c.set_option(lgc.OPT_TABLE_FORM, 2)
        ref = oracle.nibble(off, col, 3, 3, 1e-9)
        for pull in (0, 1):
            c.set_option(lgc.OPT_PULL, pull)
            for mode in ("atomic", "det"):
                p, st = lgc.nibble(g, 3, 3, 1e-9, mode=mode)
                assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes,
                                                                   ref.pushed_edges)
                assert np.array_equal(p.idx, ref.idx)
                if mode == "det":
                    assert np.array_equal(p.val, ref.val)
                else:  # three rounds; the hub's sum comes in another order
                    assert np.abs(p.val - ref.val).sum() <= 3 * (n // 16 + 1) * 2.0 ** -53
    finally:
        g.close()
        c.close()
