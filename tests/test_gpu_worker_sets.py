"""The request loop's workers hold the sets their requests were admitted by."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [14, 18])
def test_small_requests_keep_small_sets(scale):
    off, col = inputs.rmat(scale, 8, seed=1)
    deg = np.diff(off)
    x = int(np.flatnonzero(deg == 2)[0])
    ref = oracle.prnibble(off, col, x, 0.2, 0.01)
    c = lgc.Context(0)
    c.set_option(lgc.OPT_SERVE_LANE, 0)
    g = lgc.Graph(c, off, col)
    try:
        r = lgc.wait(c, lgc.submit(c, g, lgc.make_request(lgc.ALGO_PRNIBBLE, x, False, alpha=0.2,
                                                          eps=0.01, mode="det")))
        assert r["status"] == 0
        assert np.array_equal(r["idx"], ref.idx) and np.array_equal(r["val"], ref.val)
        # admitted at 24 bytes for each of 1024 slots (501 keys at most) and key
        assert 24 * r["stats"]["table_capacity"] <= 24 * 1024 + 24 * 501
    finally:
        g.close()
        c.close()
