"""Device-driven PR-Nibble rounds against the oracle: deterministic rounds bit
for bit at the sizes where the order of a destination's contributions is
found another way (by a thread, a warp, the block), beta rounds, round limits
in the middle of a launch, and the wide atomic rounds."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = lgc.Context(0)  # untraced: the device rounds run
    yield c
    c.close()


def fan(c, seed):
    """Two hubs joined through c vertices of different degrees: a push of those
    sends c different shares to each hub in one round."""
    rng = np.random.default_rng(seed)
    e = [(0, 2 + i) for i in range(c)] + [(1, 2 + i) for i in range(c)]
    n = 2 + c
    for i in range(c):
        for _ in range(int(rng.integers(0, 6))):
            e.append((2 + i, n))
            n += 1
    return inputs.from_edges(n, e)


@pytest.mark.parametrize("rule", ["opt", "orig"])
@pytest.mark.parametrize("c", [1, 7, 8, 9, 31, 32, 33, 127, 128, 129, 512, 513, 2500])
def test_det_buckets(ctx, c, rule):
    off, col = fan(c, c)
    g = lgc.Graph(ctx, off, col)
    ref = oracle.prnibble(off, col, 0, 0.05, 1e-7, rule=0 if rule == "opt" else 1)
    p, st = lgc.prnibble(g, 0, 0.05, 1e-7, rule=rule, mode="det")
    assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes, ref.pushed_edges)
    assert np.array_equal(p.idx, ref.idx) and np.array_equal(p.val, ref.val)
    g.close()


GRAPHS = {"star1500": (lambda: inputs.star(1500), 0.05, 1e-6),
          "grid17": (lambda: inputs.grid3d(17), 0.01, 1e-6),
          "rmat12": (lambda: inputs.rmat(12, seed=1), 0.01, 1e-6),
          "rmat16": (lambda: inputs.rmat(16, seed=1), 0.01, 1e-7)}


@pytest.mark.parametrize("rule", ["opt", "orig"])
@pytest.mark.parametrize("form", [0, 1, 2], ids=["auto", "hashed", "dense"])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_det_rounds(ctx, name, form, rule):
    make, alpha, eps = GRAPHS[name]
    off, col = make()
    g = lgc.Graph(ctx, off, col)
    ctx.set_option(lgc.OPT_TABLE_FORM, form)
    try:
        x = inputs.config1_seed(off, col)
        for limit in (0, 1, 6):
            ref = oracle.prnibble(off, col, x, alpha, eps, rule=0 if rule == "opt" else 1,
                                  **({"max_rounds": limit} if limit else {}))
            p, st = lgc.prnibble(g, x, alpha, eps, rule=rule, mode="det", max_rounds=limit)
            assert (st.rounds, st.pushed_edges) == (ref.rounds, ref.pushed_edges)
            assert np.array_equal(p.idx, ref.idx) and np.array_equal(p.val, ref.val)
    finally:
        ctx.set_option(lgc.OPT_TABLE_FORM, 0)
        g.close()


@pytest.mark.parametrize("mode", ["atomic", "det"])
@pytest.mark.parametrize("rule", ["opt", "orig"])
@pytest.mark.parametrize("beta", [0.9, 0.5, 0.03])
def test_beta_rounds(ctx, beta, rule, mode):
    off, col = inputs.rmat(13, seed=9)
    g = lgc.Graph(ctx, off, col)
    cand = np.flatnonzero(np.diff(off) >= 1)
    rng = np.random.default_rng(4)
    s = rng.choice(cand, size=9, replace=False).astype(np.int32)
    w = rng.uniform(0.001, 3.0, size=9)  # some seeds start below their threshold
    ref = oracle.prnibble_set(off, col, s, w, 0.05, 1e-5, rule=0 if rule == "opt" else 1, beta=beta)
    p, st = lgc.prnibble_set(g, s, 0.05, 1e-5, weights=w, beta=beta, rule=rule, mode=mode)
    assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes, ref.pushed_edges)
    assert np.array_equal(p.idx, ref.idx)
    if mode == "det":
        assert np.array_equal(p.val, ref.val)
    else:
        assert np.abs(p.val - ref.val).sum() <= 1e-12 * ref.val.sum()
    g.close()


@pytest.mark.parametrize("pull", [0, 1], ids=["wide", "plain"])
@pytest.mark.parametrize("c", [1100, 5000])
def test_hot_destinations(ctx, c, pull):
    """Frontiers of more than 2048 vertices that all push into the two hubs
    (degree 1024 and more): the hubs' adds are combined."""
    off, col = fan(c, 3)
    g = lgc.Graph(ctx, off, col)
    ctx.set_option(lgc.OPT_PULL, pull)
    try:
        for x in (0, 5):
            for ref, (p, st) in (
                    (oracle.prnibble(off, col, x, 0.05, 1e-8),
                     lgc.prnibble(g, x, 0.05, 1e-8, mode="atomic")),
                    (oracle.nibble(off, col, x, 9, 1e-9), lgc.nibble(g, x, 9, 1e-9)),
                    (oracle.hkpr(off, col, x, 4.0, 9, 1e-9), lgc.hkpr(g, x, 4.0, 9, 1e-9))):
                assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes,
                                                                   ref.pushed_edges)
                assert np.array_equal(p.idx, ref.idx)
                assert np.abs(p.val - ref.val).sum() <= 1e-12 * ref.val.sum()
    finally:
        ctx.set_option(lgc.OPT_PULL, 0)
        g.close()


FRESH = {"star1500": (lambda: inputs.star(1500), 1e-6),
         "path40": (lambda: inputs.path(40), 1e-3),
         "grid17": (lambda: inputs.grid3d(17), 1e-7),
         "rmat12": (lambda: inputs.rmat(12, seed=1), 1e-6),
         "rmat16": (lambda: inputs.rmat(16, seed=1), 1e-7)}


@pytest.mark.parametrize("mode", ["atomic", "det"])
@pytest.mark.parametrize("form", [0, 1, 2], ids=["auto", "hashed", "dense"])
@pytest.mark.parametrize("name", list(FRESH))
def test_fresh_set_rounds(ctx, name, form, mode):
    """Nibble (its early exit too) and HK-PR rounds into fresh sets."""
    make, eps = FRESH[name]
    off, col = make()
    g = lgc.Graph(ctx, off, col)
    ctx.set_option(lgc.OPT_TABLE_FORM, form)
    try:
        x = inputs.config1_seed(off, col)
        runs = []
        for T, e in ((1, eps), (2, eps), (17, eps), (25, 300 * eps), (6, 0.3), (4, 0.0)):
            runs.append((oracle.nibble(off, col, x, T, e), lgc.nibble(g, x, T, e, mode=mode)))
        for t, N, e in ((5.0, 12, eps), (5.0, 2, eps), (1.0, 1, eps), (8.0, 20, 100 * eps),
                        (2.0, 4, 0.0)):
            runs.append((oracle.hkpr(off, col, x, t, N, e), lgc.hkpr(g, x, t, N, e, mode=mode)))
        for ref, (p, st) in runs:
            assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes,
                                                               ref.pushed_edges)
            assert st.touched == ref.touched
            assert np.array_equal(p.idx, ref.idx)
            if mode == "det":
                assert np.array_equal(p.val, ref.val)
            else:
                assert np.abs(p.val - ref.val).sum() <= 1e-12 * ref.val.sum()
    finally:
        ctx.set_option(lgc.OPT_TABLE_FORM, 0)
        g.close()


def test_wide_atomic_rounds_sum_as_pull_rounds(ctx):
    """Every round of this diffusion is one that the host would run as a pull
    round: the exact sums give the same bits either way."""
    off, col = inputs.random_graph(2000, 3000, seed=8)
    hub = [(0, i) for i in range(1, 2000)]
    src = np.repeat(np.arange(2000), np.diff(off))
    off, col = inputs.from_edges(2000, list(zip(src, col)) + hub)
    g = lgc.Graph(ctx, off, col)
    out = []
    for dev in (1, 0):
        ctx.set_option(lgc.OPT_DEVICE_ROUNDS, dev)
        p, st = lgc.prnibble(g, 0, 0.2, 1e-6, mode="atomic", max_rounds=4)
        out.append((p.idx, p.val, st.pushed_edges))
    ctx.set_option(lgc.OPT_DEVICE_ROUNDS, 1)
    ref = oracle.prnibble(off, col, 0, 0.2, 1e-6, max_rounds=4)
    assert out[0][2] == out[1][2] == ref.pushed_edges
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    g.close()
