"""Hashed sets of the device rounds past the slots they get ahead of need."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import lgc

pytestmark = pytest.mark.gpu


def tassels(n, step):
    """Vertex 0 joined to every step-th vertex, each of which to its successor."""
    leaf = np.arange(step, n - 1, step, dtype=np.int64)
    a = np.concatenate([np.zeros_like(leaf), leaf, leaf, leaf + 1])
    b = np.concatenate([leaf, np.zeros_like(leaf), leaf + 1, leaf])
    order = np.lexsort((b, a))
    off = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(a, minlength=n), out=off[1:])
    return off, b[order].astype(np.int32)


@pytest.mark.parametrize("mode", ["det", "atomic"])
@pytest.mark.parametrize("n,step", [(8_000_000, 27), (5_000_000, 9)])
def test_past_the_room_ahead(n, step, mode):
    off, col = tassels(n, step)
    leaves = int(off[1])
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        c.set_option(lgc.OPT_TABLE_FORM, 1)
        for ref, (p, st) in (
                (oracle.prnibble(off, col, step, 0.05, 1e-8),
                 lgc.prnibble(g, step, 0.05, 1e-8, mode=mode)),
                (oracle.nibble(off, col, step, 6, 1e-9), lgc.nibble(g, step, 6, 1e-9, mode=mode)),
                (oracle.hkpr(off, col, step, 3.0, 6, 1e-9),
                 lgc.hkpr(g, step, 3.0, 6, 1e-9, mode=mode))):
            assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes,
                                                               ref.pushed_edges)
            assert np.array_equal(p.idx, ref.idx)
            if mode == "det":
                assert np.array_equal(p.val, ref.val)
            else:  # the hub's sums come in another order, once a round
                assert (np.abs(p.val - ref.val).sum()
                        <= ref.rounds * leaves * 2.0 ** -53 * ref.val.sum())
    finally:
        g.close()
        c.close()
