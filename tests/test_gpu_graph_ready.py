"""A graph's lists are complete when the call that builds them returns: the
request loop and other contexts read them on streams of their own."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu

GRAPHS = {"grid9": lambda: inputs.grid3d(9), "star1500": lambda: inputs.star(1500),
          "rmat12": lambda: inputs.rmat(12, seed=1), "no_edges": lambda: inputs.from_edges(40, [])}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_nothing_in_flight(name):
    """Every allocation puts a millisecond of work on the stream, so work that a
    call leaves behind is still there when it returns."""
    import torch
    off, col = GRAPHS[name]()
    s = torch.cuda.Stream()

    def alloc(nbytes, stream):
        with torch.cuda.stream(s):
            torch.cuda._sleep(2_000_000)
        return torch.cuda.caching_allocator_alloc(nbytes, 0, stream)

    c = lgc.Context(0, s, allocator=(alloc, lambda ptr, st: torch.cuda.caching_allocator_delete(ptr)))
    try:
        g = lgc.Graph(c, off, col)
        assert s.query()
        for light in (4, 64, 32):
            g.set_pull_light(light)
            assert s.query()
        g.close()
    finally:
        c.close()


@pytest.mark.parametrize("name", ["grid9", "rmat12"])
def test_submit_at_once(name):
    off, col = GRAPHS[name]()
    x = inputs.config1_seed(off, col)
    ref = oracle.prnibble(off, col, x, 0.05, 1e-5)
    rs = oracle.sweep(off, col, ref.idx, ref.val)
    hk = oracle.hkpr(off, col, x, 4.0, 10, 1e-5)
    c = lgc.Context(0)
    for light in (0, 4, 128):
        g = lgc.Graph(c, off, col)
        if light:
            g.set_pull_light(light)
        t = [lgc.submit(c, g, lgc.make_request(lgc.ALGO_PRNIBBLE, x, True, alpha=0.05, eps=1e-5,
                                               mode="det")),
             lgc.submit(c, g, lgc.make_request(lgc.ALGO_HKPR, x, True, t=4.0, N=10, eps=1e-5,
                                               mode="det"))]
        a, b = [lgc.wait(c, k) for k in t]
        assert np.array_equal(a["idx"], ref.idx) and np.array_equal(a["val"], ref.val)
        assert (a["cluster"]["vol"], a["cluster"]["cut"]) == (rs.best_vol, rs.best_cut)
        assert np.array_equal(b["idx"], hk.idx) and np.array_equal(b["val"], hk.val)
        g.close()
    c.close()
