"""CSRs that LGC_GRAPH_VALIDATE would refuse but that are taken without it:
one-way edges (more edges into a vertex than it has itself), repeated edges,
lists in any order.  Deterministic pushes follow the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1604_07515_gb300 import inputs, lgc

pytestmark = pytest.mark.gpu


def csr(lists):
    off = np.zeros(len(lists) + 1, np.int64)
    np.cumsum([len(a) for a in lists], out=off[1:])
    return off, np.concatenate([np.asarray(a, np.int32) for a in lists]).astype(np.int32)


def into_few(n, heads, rng):
    """Every vertex points to all of the first few, those back to a handful."""
    out = [sorted(rng.choice(np.arange(heads, n), size=3, replace=False)) for _ in range(heads)]
    for v in range(heads, n):
        out.append(list(range(heads)) + [heads + (v - heads + 1) % (n - heads)])
    return csr(out)


def one_way(n, rng):
    return csr([sorted(rng.choice(n, size=int(rng.integers(1, 9)), replace=False))
                for _ in range(n)])


def repeated(n, rng):
    """Symmetric, every edge one to four times."""
    lists = [[] for _ in range(n)]
    for v in range(n):
        for u in rng.choice(n, size=4, replace=False):
            if u != v:
                for _ in range(int(rng.integers(1, 5))):
                    lists[v].append(int(u))
                    lists[u].append(v)
    return csr([sorted(a) for a in lists])


def shuffled(n, rng):
    off, col = inputs.random_graph(n, 4 * n, seed=n)
    col = col.copy()
    for v in range(n):
        rng.shuffle(col[off[v]:off[v + 1]])
    return off, col


def make(name):
    rng = np.random.default_rng(len(name))
    return {"into3": lambda: into_few(3000, 3, rng), "into40": lambda: into_few(700, 40, rng),
            "one_way": lambda: one_way(2000, rng), "repeated": lambda: repeated(600, rng),
            "hub_repeated": lambda: csr([list(np.repeat(np.arange(1, 200), 3))] +
                                        [[0] * 3 + [1 + v % 199] * 2 for v in range(1, 200)]),
            "shuffled": lambda: shuffled(900, rng)}[name]()


@pytest.mark.parametrize("name", ["into3", "into40", "one_way", "repeated", "hub_repeated",
                                  "shuffled"])
def test_det_pushes(name):
    off, col = make(name)
    x = 1
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        c.set_option(lgc.OPT_PULL, 1)  # gathers would read the lists the other way round
        s = np.array([1, 5, 7], np.int32)
        w = np.array([1.0, 0.3, 2.0])
        for ref, (p, st) in (
                (oracle.prnibble(off, col, x, 0.05, 1e-6),
                 lgc.prnibble(g, x, 0.05, 1e-6, mode="det")),
                (oracle.prnibble_set(off, col, s, w, 0.05, 1e-5, rule=1, beta=0.5),
                 lgc.prnibble_set(g, s, 0.05, 1e-5, weights=w, beta=0.5, rule="orig", mode="det")),
                (oracle.nibble(off, col, x, 12, 1e-7), lgc.nibble(g, x, 12, 1e-7, mode="det")),
                (oracle.hkpr(off, col, x, 4.0, 9, 1e-7), lgc.hkpr(g, x, 4.0, 9, 1e-7, mode="det"))):
            assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes,
                                                               ref.pushed_edges)
            assert np.array_equal(p.idx, ref.idx) and np.array_equal(p.val, ref.val)
    finally:
        g.close()
        c.close()


def sinks(n, out, deg, seed):
    """Vertices below `out` point anywhere (vertex 1 to half of all), the others
    nowhere."""
    rng = np.random.default_rng(seed)
    size = rng.integers(1, deg + 1, size=out)
    size[1] = n // 2
    return csr([sorted(rng.choice(n, size=int(size[v]), replace=False)) if v < out else []
                for v in range(n)])


@pytest.mark.parametrize("form", [0, 1, 2], ids=["auto", "hashed", "dense"])
@pytest.mark.parametrize("device", [1, 0])
@pytest.mark.parametrize("n,out,deg", [(3000, 1500, 8), (4000, 400, 300), (900, 600, 1),
                                       (2500, 40, 2000)])
def test_vertices_without_edges(n, out, deg, device, form):
    """Frontiers in which many vertices in a row have no edges."""
    off, col = sinks(n, out, deg, n)
    c = lgc.Context(0)
    g = lgc.Graph(c, off, col)
    try:
        c.set_option(lgc.OPT_PULL, 1)
        c.set_option(lgc.OPT_DEVICE_ROUNDS, device)
        c.set_option(lgc.OPT_TABLE_FORM, form)
        for mode in ("det", "atomic"):
            for ref, (p, st) in (
                    (oracle.nibble(off, col, 1, 5, 0.0), lgc.nibble(g, 1, 5, 0.0, mode=mode)),
                    (oracle.hkpr(off, col, 1, 3.0, 6, 0.0),
                     lgc.hkpr(g, 1, 3.0, 6, 0.0, mode=mode))):
                assert (st.rounds, st.pushes, st.pushed_edges) == (ref.rounds, ref.pushes,
                                                                   ref.pushed_edges)
                assert np.array_equal(p.idx, ref.idx)
                if mode == "det":
                    assert np.array_equal(p.val, ref.val)
                else:  # at most 6 rounds whose sums of up to `out` terms come in another order
                    assert np.abs(p.val - ref.val).sum() <= 6 * out * 2.0 ** -53 * ref.val.sum()
    finally:
        g.close()
        c.close()
