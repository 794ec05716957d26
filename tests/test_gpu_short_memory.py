"""Calls on a device with little memory left: what the device rounds and the
graph's tables would like is given up where it cannot be had, and the
host-driven rounds, divisions and plain pushes give the same results."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


class Memory:
    """Device memory that refuses what `refuse(nbytes)` says."""

    def __init__(self):
        self.refuse = lambda nbytes: False
        self.most, self.refused, self.live = 0, 0, {}

    def alloc(self, nbytes, stream):
        import torch
        if self.refuse(nbytes):
            self.refused += 1
            return 0
        self.most = max(self.most, nbytes)
        ptr = torch.cuda.caching_allocator_alloc(nbytes, 0, stream)
        self.live[ptr] = nbytes
        return ptr

    def free(self, ptr, stream):
        import torch
        del self.live[ptr]
        torch.cuda.caching_allocator_delete(ptr)


def calls(g, off, col, x, eps, mode):
    """(oracle, library) results of one call of each diffusion."""
    s = np.array([x, x + 1], np.int32)
    # (a selection among candidates that only rounding tells apart, as on a
    # mesh, is the oracle's in deterministic mode only)
    beta = 0.5 if mode == "det" else 1.0
    return [(lambda: oracle.prnibble(off, col, x, 0.05, eps),
             lambda: lgc.prnibble(g, x, 0.05, eps, mode=mode)),
            (lambda: oracle.prnibble_set(off, col, s, [1.0, 2.0], 0.05, eps, beta=beta),
             lambda: lgc.prnibble_set(g, s, 0.05, eps, weights=[1.0, 2.0], beta=beta, mode=mode)),
            (lambda: oracle.nibble(off, col, x, 9, eps),
             lambda: lgc.nibble(g, x, 9, eps, mode=mode)),
            (lambda: oracle.hkpr(off, col, x, 3.0, 9, eps),
             lambda: lgc.hkpr(g, x, 3.0, 9, eps, mode=mode))]


def same(ref, got, mode):
    p, st = got
    assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes, ref.pushed_edges)
    assert np.array_equal(p.idx, ref.idx)
    if mode == "det":
        assert np.array_equal(p.val, ref.val)
    else:
        assert np.abs(p.val - ref.val).sum() <= 1e-12 * ref.val.sum()


@pytest.mark.parametrize("form", [0, 1], ids=["auto", "hashed"])
@pytest.mark.parametrize("mode", ["det", "atomic"])
def test_room_for_host_rounds_only(mode, form):
    """No request above the largest of the host-driven call is met."""
    off, col = inputs.grid3d(40)
    m = Memory()
    c = lgc.Context(0, allocator=(m.alloc, m.free))
    g = lgc.Graph(c, off, col)
    c.set_option(lgc.OPT_TABLE_FORM, form)
    for ref, call in calls(g, off, col, 777, 1e-5, mode):
        ref = ref()
        c.set_option(lgc.OPT_DEVICE_ROUNDS, 0)
        m.most = m.refused = 0
        same(ref, call(), mode)
        limit = m.most
        c.set_option(lgc.OPT_DEVICE_ROUNDS, 1)
        m.refuse = lambda nbytes: nbytes > limit
        same(ref, call(), mode)
        assert m.refused > 0
        m.refuse = lambda nbytes: False
        same(ref, call(), mode)
    g.close()
    c.close()
    assert not m.live


@pytest.mark.parametrize("which", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("mode", ["det", "atomic"])
def test_one_of_the_large_requests(mode, which):
    """One of the requests above the host-driven call's largest is refused: the
    buckets, the slab, the per-slot array or a set."""
    off, col = inputs.grid3d(40)
    m = Memory()
    c = lgc.Context(0, allocator=(m.alloc, m.free))
    g = lgc.Graph(c, off, col)
    for ref, call in calls(g, off, col, 777, 1e-5, mode):
        ref = ref()
        c.set_option(lgc.OPT_DEVICE_ROUNDS, 0)
        m.most = 0
        same(ref, call(), mode)
        limit, seen = m.most, []
        c.set_option(lgc.OPT_DEVICE_ROUNDS, 1)

        def refuse(nbytes):
            if nbytes > limit:
                seen.append(nbytes)
                return len(seen) == which + 1
            return False

        m.refuse = refuse
        same(ref, call(), mode)
        m.refuse = lambda nbytes: False
    g.close()
    c.close()
    assert not m.live


def test_graph_without_its_tables():
    """The reciprocals, the hot vertices' table and the entry counts refused."""
    off, col = inputs.star(1500)
    for size in (16 * (int(np.diff(off).max()) + 1), 512 + 8 * 16384, 8 * (256 + 32),
                 32 + 4 * (len(off) - 1)):
        m = Memory()
        m.refuse = lambda nbytes: nbytes == size
        c = lgc.Context(0, allocator=(m.alloc, m.free))
        g = lgc.Graph(c, off, col)
        assert m.refused == 1
        for mode in ("det", "atomic"):
            for ref, call in calls(g, off, col, 0, 1e-6, mode):
                same(ref(), call(), mode)
        ref = oracle.prnibble(off, col, 0, 0.05, 1e-6)
        rs = oracle.sweep(off, col, ref.idx, ref.val)
        p, _ = lgc.prnibble(g, 0, 0.05, 1e-6, mode="det")
        k = lgc.sweep(g, p)
        assert (k.size, k.vol, k.cut) == (rs.best, rs.best_vol, rs.best_cut)
        del p, k
        g.close()
        c.close()
        assert not m.live
