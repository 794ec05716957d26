"""Host-driven gathers at the degree bins' edges in the forms that a large graph
or a full device gets: without interleaved columns, and deterministic long
lists without kept shares."""
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


def slice_bytes(off):
    d = np.diff(off)
    d = np.sort(d[(d >= 1) & (d <= 1024)])[::-1]
    return 4 * 32 * int(d[::32].sum())


def kept_bytes(off):
    d = np.diff(off)
    shares, cap = 256 * int((-(-d[d > 1024] // 256)).sum()), 1024
    while cap < shares:
        cap *= 2
    return 8 * cap


# (requests are told by their size: one segment's shares are as large as others)
@pytest.mark.parametrize("without,count", [("nothing", 1), ("nothing", 33), ("slices", 1),
                                           ("slices", 33), ("kept", 33), ("kept", 70)])
def test_gathers(without, count):
    import torch
    off, col = binned(count)
    size = {"nothing": -1, "slices": slice_bytes(off), "kept": kept_bytes(off)}[without]
    refused = []

    def alloc(nbytes, stream):
        if nbytes == size:
            refused.append(nbytes)
            return 0
        return torch.cuda.caching_allocator_alloc(nbytes, 0, stream)

    c = lgc.Context(0, allocator=(alloc,
                                  lambda p, s: torch.cuda.caching_allocator_delete(p)))
    g = lgc.Graph(c, off, col)
    try:
        c.set_option(lgc.OPT_PULL, 2)
        c.set_option(lgc.OPT_DEVICE_ROUNDS, 0)
        c.set_option(lgc.OPT_SWEEP_CROSS, 2)
        terms = int(np.diff(off).max()) + 2
        for eps in (1e-7, 1e-4, 0.0):
            ref = oracle.hkpr(off, col, 5, 5.0, 8, eps)
            for light in (4, 32, 256):
                g.set_pull_light(light)
                for share in (8, 16):
                    c.set_option(lgc.OPT_PULL_SHARE, share)
                    for mode in ("det", "atomic"):
                        p, st = lgc.hkpr(g, 5, 5.0, 8, eps, mode=mode)
                        assert (st.rounds, st.pushes, st.pushed_edges) == (
                            ref.rounds, ref.pushes, ref.pushed_edges)
                        assert np.array_equal(p.idx, ref.idx)
                        if mode == "det":
                            assert np.array_equal(p.val, ref.val)
                        else:  # sums rounded once here, once a term in the oracle
                            assert (np.abs(p.val - ref.val).sum()
                                    <= 8 * terms * 2.0 ** -53 * ref.val.sum())
        ref = oracle.prnibble(off, col, 5, 0.05, 1e-6)
        p, st = lgc.prnibble(g, 5, 0.05, 1e-6, mode="det")
        assert np.array_equal(p.idx, ref.idx) and np.array_equal(p.val, ref.val)
        rs = oracle.sweep(off, col, ref.idx, ref.val)
        k = lgc.sweep(g, p)
        assert (k.size, k.vol, k.cut) == (rs.best, rs.best_vol, rs.best_cut)
        assert np.array_equal(k.ids, rs.cluster)
        assert bool(refused) == (without != "nothing")
        del p, k
    finally:
        g.close()
        c.close()
