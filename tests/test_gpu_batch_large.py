"""Batches whose results are large enough to be copied one by one, and rounds
whose warps cross from seed to seed at the hub."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 2, 33])
@pytest.mark.parametrize("mode", ["det", "atomic"])
def test_large_results(B, mode):
    off, col = inputs.rmat(16, seed=1)
    rng = np.random.default_rng(B)
    seeds = rng.choice(np.flatnonzero(np.diff(off) >= 2), B, replace=False).astype(np.int32)
    eps = np.full(B, 2e-7)
    eps[B // 2:] *= 0.5
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        ps, sts = lgc.prnibble_batch(g, seeds, 0.01, eps, rule="opt", mode=mode)
        assert sum(p.nnz for p in ps) >= 4096 * B
        cs = lgc.sweep_batch(g, ps)
        for b in range(0, B, 11):
            ref = oracle.prnibble(off, col, int(seeds[b]), 0.01, eps[b])
            if mode == "det":
                assert np.array_equal(ps[b].idx, ref.idx) and np.array_equal(ps[b].val, ref.val)
                assert sts[b].pushed_edges == ref.pushed_edges
            else:  # as the single-seed atomic mode's tests
                p = np.zeros(len(off) - 1)
                p[ps[b].idx] = ps[b].val
                p[ref.idx] -= ref.val
                assert np.abs(p).sum() <= 1e-12 * ref.val.sum()
            one = lgc.sweep(g, ps[b])
            assert (cs[b].size, cs[b].vol, cs[b].cut) == (one.size, one.vol, one.cut)
            assert np.array_equal(cs[b].ids, one.ids)
    finally:
        g.close()
        c.close()
