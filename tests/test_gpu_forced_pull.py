"""LGC_OPT_PULL = 2: every round of HK-PR gathers, in atomic mode too, whose
gathers round each sum once, so the device rounds' option changes no bit."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("light", [4, 32, 256])
@pytest.mark.parametrize("n,m,hubs", [(900, 4000, 3), (3001, 9000, 1), (5000, 30000, 2)])
def test_forced_pull_atomic_hkpr(n, m, hubs, light):
    off, col = inputs.random_graph(n, m, seed=n)
    src = np.repeat(np.arange(n), np.diff(off))
    e = [(h, v) for h in range(hubs) for v in range(hubs, n, h + 1)]
    off, col = inputs.from_edges(n, list(zip(src, col)) + e)
    ref = oracle.hkpr(off, col, n - 1, 6.0, 12, 1e-9)
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        g.set_pull_light(light)
        c.set_option(lgc.OPT_PULL, 2)
        got = []
        for device in (1, 0):
            c.set_option(lgc.OPT_DEVICE_ROUNDS, device)
            p, st = lgc.hkpr(g, n - 1, 6.0, 12, 1e-9, mode="atomic")
            assert (st.rounds, st.pushed_edges) == (ref.rounds, ref.pushed_edges)
            got.append((p.idx.copy(), p.val.copy()))
        assert np.array_equal(got[0][0], ref.idx) and np.array_equal(got[1][0], ref.idx)
        assert np.array_equal(got[0][1], got[1][1])
        # a round's sums are rounded once here and once per term in the oracle
        terms = int(np.diff(off).max()) + 2
        assert np.abs(got[1][1] - ref.val).sum() <= 12 * terms * 2.0 ** -53 * ref.val.sum()
    finally:
        g.close()
        c.close()
