"""Admission counts the shares that deterministic gathers keep."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


def hubs(k, n):
    """k vertices joined to all others."""
    return inputs.from_edges(n, [(h, v) for h in range(k) for v in range(k, n)])


@pytest.mark.parametrize("algo", ["hkpr", "nibble"])
def test_one_at_a_time(algo):
    """40 lists of 2960: 480 segments' shares take 1 MB, the sets 0.12 MB.  With
    a budget of 0.5 MB no two requests are in flight together."""
    off, col = hubs(40, 3000)
    c = lgc.Context(0)
    c.set_option(lgc.OPT_SERVE_MEM_BUDGET, 500_000)
    g = lgc.Graph(c, off, col)
    try:
        if algo == "hkpr":
            ref = oracle.hkpr(off, col, 50, 5.0, 20, 1e-9)
            req = lgc.make_request(lgc.ALGO_HKPR, 50, False, t=5.0, N=20, eps=1e-9, mode="det")
        else:
            ref = oracle.nibble(off, col, 50, 20, 1e-9)
            req = lgc.make_request(lgc.ALGO_NIBBLE, 50, False, T=20, eps=1e-9, mode="det")
        got = [lgc.wait(c, t) for t in [lgc.submit(c, g, req) for _ in range(8)]]
        for r in got:
            assert r["status"] == 0
            assert np.array_equal(r["idx"], ref.idx) and np.array_equal(r["val"], ref.val)
        got.sort(key=lambda r: r["start_s"])
        assert all(b["start_s"] >= a["end_s"] for a, b in zip(got, got[1:]))
    finally:
        g.close()
        c.close()
