"""The work this library is measured on: calls as a user's program makes them.

Every case builds its graph on the GPU from the seed (R-MAT with the
partition probabilities 0.57, 0.19, 0.19, 0.05, or the 3-D torus), keeps a
context and a graph handle as a program does, and times whole calls through
the Python binding with the default host results: a diffusion and the sweep
cut of its vector, a batch of seeds with its sweeps, or a burst of requests.

A case is a dict of plain values:

* ``kind``: prnibble, set (weighted seed set with beta-fraction rounds),
  nibble, hkpr, rand_hkpr, batch (many seeds in one call) or serve (requests
  through the request loop);
* ``n``, ``ef``: vertices and sampled edges per vertex of the R-MAT graph
  (``ef`` 0: the torus of side round(n ** (1/3)));
* ``start``: "hub" (the highest-degree neighbour of vertex 0) or "any" (a
  vertex of degree >= 2);
* ``mode``: "atomic" or "det"; ``tuned``: whether the program calls
  ``autotune()`` once on its graph;
* the method's parameters (alpha, eps, rule, T, t, N, K, walks, B, k, beta).
"""
import math

import numpy as np
import torch

from paper_1604_07515_gb300 import lgc


def listed():
    return [
        # the smallest call: a query on a graph that fits in cache, where
        # launches and round trips are all there is
        dict(name="prnibble_small", kind="prnibble", n=1 << 12, ef=16, start="hub", mode="det",
             rule="opt", alpha=0.01, eps=1e-5),
        # one interactive query on a small social graph
        dict(name="prnibble_16", kind="prnibble", n=1 << 16, ef=16, start="hub", mode="atomic",
             rule="opt", alpha=0.01, eps=1e-6),
        # a weighted seed set, half of the candidates pushed per round, on a
        # graph whose size is no power of two
        dict(name="prnibble_set", kind="set", n=262_139, ef=16, start="any", mode="atomic",
             rule="orig", alpha=0.05, eps=1e-6, k=16, beta=0.5),
        # a mesh: every degree 6, many rounds of small frontiers
        dict(name="prnibble_torus", kind="prnibble", n=60 ** 3, ef=0, start="any", mode="det",
             rule="opt", alpha=0.01, eps=1e-6),
        # one query that reaches much of a large graph
        dict(name="prnibble_22", kind="prnibble", n=1 << 22, ef=16, start="hub", mode="atomic",
             rule="opt", alpha=0.01, eps=1e-7),
        # the same call where results have to be reproducible bit for bit, at
        # the finest threshold in use
        dict(name="prnibble_24_det", kind="prnibble", n=1 << 24, ef=16, start="any", mode="det",
             rule="opt", alpha=0.01, eps=1e-8),
        # truncated lazy walks: a fresh vector every step
        dict(name="nibble_22", kind="nibble", n=1 << 22, ef=16, start="hub", mode="atomic",
             T=20, eps=1e-8),
        # heat kernel over the whole graph on a tuned handle: the gathers
        # carry it
        dict(name="hkpr_22", kind="hkpr", n=1 << 22, ef=16, start="hub", mode="atomic",
             tuned=True, t=10.0, N=20, eps=1e-7),
        # the same reproducibly, on a ragged graph with another density
        dict(name="hkpr_det", kind="hkpr", n=1_500_007, ef=12, start="hub", mode="det",
             tuned=False, t=10.0, N=20, eps=1e-7),
        # Monte Carlo heat kernel
        dict(name="rand_hkpr_22", kind="rand_hkpr", n=1 << 22, ef=16, start="hub", t=10.0, K=10,
             walks=1_000_000),
        # many seeds in one call, thresholds spread over three decades
        dict(name="batch_1024", kind="batch", n=1 << 24, ef=16, start="any", mode="atomic",
             rule="opt", alpha=0.01, eps=1e-8, B=1024),
        # a burst of requests, four PR-Nibble to one HK-PR, through the
        # request loop
        dict(name="serve_burst", kind="serve", n=1 << 20, ef=16, start="any", mode="atomic",
             alpha=0.01, eps=1e-8, B=20),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["prnibble", "prnibble", "prnibble", "set", "nibble", "nibble", "hkpr",
                       "hkpr", "hkpr", "rand_hkpr", "batch", "serve"])
    top = {"serve": 1 << 20, "batch": 1 << 23}.get(kind, 1 << 22)
    n = int(_log(rng, 1 << 12, top)) | rng.randrange(2)
    c = dict(kind=kind, n=n, ef=rng.randrange(6, 21), start=rng.choice(["hub", "any"]))
    if kind in ("prnibble", "set", "batch"):
        c.update(mode=rng.choice(["atomic", "det"]), rule=rng.choice(["opt", "opt", "orig"]),
                 alpha=round(_log(rng, 0.005, 0.1), 4), eps=float("%.2g" % _log(rng, 1e-8, 1e-5)))
        if kind == "prnibble" and rng.random() < 0.25:
            c.update(n=int(round(n ** (1 / 3))) ** 3, ef=0, start="any", mode="det",
                     eps=max(c["eps"], 1e-7))
        if kind == "set":
            c.update(k=rng.randrange(2, 64), beta=round(rng.uniform(0.2, 1.0), 2), start="any",
                     eps=max(c["eps"], 1e-7))
        if kind == "batch":
            c.update(B=int(_log(rng, 8, 512)), start="any")
    elif kind == "nibble":
        c.update(mode=rng.choice(["atomic", "det"]), T=rng.randrange(5, 31),
                 eps=float("%.2g" % _log(rng, 1e-8, 1e-5)))
    elif kind == "hkpr":
        c.update(mode=rng.choice(["atomic", "atomic", "det"]), tuned=rng.random() < 0.3,
                 t=round(_log(rng, 3.0, 20.0), 2), N=rng.randrange(8, 31),
                 eps=float("%.2g" % _log(rng, 1e-8, 1e-5)))
    elif kind == "rand_hkpr":
        c.update(t=round(_log(rng, 3.0, 20.0), 2), K=rng.randrange(4, 31),
                 walks=int(_log(rng, 10_000, 4_000_000)))
    else:
        c.update(mode="atomic", alpha=0.01, eps=1e-8, B=rng.randrange(5, 21), start="any")
    return c


# ---- inputs ----

def _rmat(n, ef, gen):
    """CSR (int64 offsets, int32 columns, on the GPU) of a symmetrised R-MAT
    graph: ef * n samples over the next power of two, those outside [0, n)
    dropped with self loops and repeats."""
    m = ef * n
    src = torch.zeros(m, dtype=torch.int32, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(max(1, (n - 1).bit_length())):
        u = torch.rand(m, generator=gen, device="cuda")
        # quadrants a 0.57, b 0.19 (right), c 0.19 (down), d 0.05 (both)
        src.mul_(2).add_((u >= 0.76).int())
        dst.mul_(2).add_(((u >= 0.57) & (u < 0.76) | (u >= 0.95)).int())
    del u
    keep = (src < n) & (dst < n) & (src != dst)
    src, dst = src[keep].long(), dst[keep].long()
    del keep
    key = torch.cat([src * n + dst, dst * n + src])
    del src, dst
    key = torch.unique(key)
    deg = torch.bincount(key // n, minlength=n)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=off[1:])
    return off, (key % n).int()


def _torus(side):
    v = torch.arange(side ** 3, device="cuda")
    x, y, z = v // (side * side), v // side % side, v % side
    nb = [((x + a) % side * side + (y + b) % side) * side + (z + c) % side
          for a, b, c in ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1))]
    col = torch.stack(nb, 1).sort(1).values
    return torch.arange(side ** 3 + 1, device="cuda") * 6, col.reshape(-1).int()


def _count(case):
    """How many start vertices the case's call takes."""
    return {"set": case.get("k"), "batch": case.get("B"), "serve": case.get("B")}.get(
        case["kind"]) or 1


def _inputs(case, seed):
    """The graph, start vertices and random parameters of (case, seed)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["ef"]:
        off, col = _rmat(case["n"], case["ef"], gen)
    else:
        off, col = _torus(int(round(case["n"] ** (1 / 3))))
    deg = off[1:] - off[:-1]
    rng = np.random.default_rng(seed)
    if case["start"] == "hub":
        nb = col[: int(off[1])].long()
        d = deg[nb]
        starts = nb[d == d.max()][:1].cpu().numpy()
    else:
        some = torch.nonzero(deg >= 2).reshape(-1)
        at = rng.choice(len(some), _count(case), replace=False)
        starts = some[torch.from_numpy(at).cuda()].cpu().numpy()
    more = {}
    if case["kind"] == "set":
        more["weights"] = rng.uniform(0.5, 2.0, len(starts))
    if case["kind"] in ("batch", "serve"):
        lo = math.log10(case["eps"])
        more["eps"] = 10.0 ** rng.uniform(lo, lo + 3.0, len(starts))
    if case["kind"] == "serve":
        more["t"] = 3.0 * 10.0 ** rng.uniform(0.0, 1.0, len(starts))
    if case["kind"] == "rand_hkpr":
        more["rng_seed"] = int(rng.integers(1 << 62))
    return off, col, starts.astype(np.int32), more


def _taylor(t):
    """Taylor terms until the Poisson tail is below 1e-6."""
    term = total = math.exp(-t)
    k = 0
    while 1.0 - total > 1e-6 and k < 200:
        k += 1
        term *= t / k
        total += term
    return max(2, k)


def prepare(case, seed):
    off, col, starts, more = _inputs(case, seed)
    torch.cuda.synchronize()  # the library works on a stream of its own
    ctx = lgc.Context(0)
    g = lgc.Graph(ctx, off, col)
    ctx.synchronize()
    if case.get("tuned"):
        g.autotune()
    s = dict(case=case, ctx=ctx, g=g, starts=starts, out={}, **more)
    if case["kind"] == "serve":
        s["requests"] = [
            lgc.make_request(lgc.ALGO_HKPR, int(x), True, t=float(s["t"][i]),
                             N=_taylor(float(s["t"][i])), eps=1e-7, mode=case["mode"])
            if i % 5 == 4 else
            lgc.make_request(lgc.ALGO_PRNIBBLE, int(x), True, alpha=case["alpha"],
                             eps=float(s["eps"][i]), mode=case["mode"])
            for i, x in enumerate(starts)]
    return s


# ---- the calls ----

def _room(case):
    """Entries that the case's sparse vectors may have together."""
    return min(case["n"] * (case["B"] if case["kind"] == "batch" else 1),
               1 << (26 if case["kind"] == "batch" else 22))


def _kept(s, name, arrays, dtype):
    """The arrays one after another at the front of a buffer that the state
    keeps; what lies behind stays zero.  Large ones are copied by torch, on
    several cores."""
    buf = s["out"].get(name)
    if buf is None:
        buf = s["out"][name] = np.zeros(_room(s["case"]), dtype)
    at = 0
    for a in arrays:
        if len(a) < 200_000:
            buf[at:at + len(a)] = a
        else:
            torch.from_numpy(buf[at:at + len(a)]).copy_(torch.from_numpy(a))
        at += len(a)
    return buf


def _cluster(s, c, mode):
    """A cluster's numbers; its members too in deterministic mode (in atomic
    mode vertices whose p/d differ only by rounding may swap places)."""
    d = dict(whole=np.array([c.size, c.vol, c.cut]), conductance=float(c.conductance))
    if mode == "det":
        d["ids"] = _kept(s, "ids", [c.ids], np.int32)
    return d


def run(s):
    """One call, its sparse results as (number of entries, ids, values) with
    room behind the entries."""
    c, g = s["case"], s["g"]
    kind, mode, x = c["kind"], c.get("mode", "det"), int(s["starts"][0])
    if kind == "batch":
        ps, _ = lgc.prnibble_batch(g, s["starts"], c["alpha"], s["eps"], rule=c["rule"], mode=mode)
        cs = lgc.sweep_batch(g, ps)
        return dict(nnz=np.array([p.nnz for p in ps]),
                    idx=_kept(s, "idx", [p.idx for p in ps], np.int32),
                    val=_kept(s, "val", [p.val for p in ps], np.float64),
                    conductance=np.array([k.conductance for k in cs]))
    if kind == "serve":
        tickets = [lgc.submit(s["ctx"], g, r) for r in s["requests"]]
        got = [lgc.wait(s["ctx"], t) for t in tickets]
        return [(_kept(s, "idx%d" % i, [r["idx"]], np.int32),
                 _kept(s, "val%d" % i, [r["val"]], np.float64),
                 float(r["cluster"]["conductance"])) for i, r in enumerate(got)]
    if kind == "prnibble":
        p, _ = lgc.prnibble(g, x, c["alpha"], c["eps"], rule=c["rule"], mode=mode)
    elif kind == "set":
        p, _ = lgc.prnibble_set(g, s["starts"], c["alpha"], c["eps"], weights=s["weights"],
                                beta=c["beta"], rule=c["rule"], mode=mode)
    elif kind == "nibble":
        p, _ = lgc.nibble(g, x, c["T"], c["eps"], mode=mode)
    elif kind == "hkpr":
        p, _ = lgc.hkpr(g, x, c["t"], c["N"], c["eps"], mode=mode)
    else:
        p, _ = lgc.rand_hkpr(g, x, c["t"], c["K"], c["walks"], s["rng_seed"])
    k = lgc.sweep(g, p)
    return dict(nnz=p.nnz, idx=_kept(s, "idx", [p.idx], np.int32),
                val=_kept(s, "val", [p.val], np.float64), cluster=_cluster(s, k, mode))


# ---- what a pass cannot do without ----

def work(case):
    """Bytes: the offset, degree and columns of every vertex that pushes or
    is swept, read once, and the results written once; flops: one add per
    pushed edge and two operations per push.  How far a diffusion spreads
    depends on the graph: the counts are those typical of these graphs."""
    nnz = case["n"] * (1.9 * case["ef"] if case["ef"] else 6)
    live = case["n"] * (0.57 if case["ef"] else 1.0)
    kind = case["kind"]

    def pr(alpha, eps):
        # the bound is 1 / (alpha eps) pushed edges
        edges = min(20 * nnz, 0.2 / (alpha * eps)) if eps * nnz < 2 else 0.005 / (alpha * eps)
        return edges, min(nnz, edges / 2), min(live, edges / 60)

    def hk(t, N, eps):
        part = min(1.0, 2.0 * N / (eps * nnz))
        return min(N, t + 3) * nnz * part, nnz * part, live * part

    if kind in ("prnibble", "set"):
        parts = [pr(case["alpha"], case["eps"])]
    elif kind == "batch":
        parts = [pr(case["alpha"], case["eps"] * 10.0 ** (3.0 * (i + 0.5) / case["B"]))
                 for i in range(case["B"])]
    elif kind == "serve":
        parts = [hk(3.0 * 10.0 ** 0.5, 20, 1e-7) if i % 5 == 4 else
                 pr(case["alpha"], case["eps"] * 10.0 ** (3.0 * (i + 0.5) / case["B"]))
                 for i in range(case["B"])]
    elif kind == "nibble":
        edges = min(case["T"] * nnz, case["T"] * 0.01 / case["eps"])
        parts = [(edges, min(nnz, edges / 4), min(live, edges / 1000))]
    elif kind == "hkpr":
        parts = [hk(case["t"], case["N"], case["eps"])]
    else:
        steps = case["walks"] * min(case["t"], case["K"])
        parts = [(steps, min(nnz, 2 * steps), min(live, case["walks"] / 3))]
    return {"bytes": sum(4 * e + (16 + 12) * v for _, e, v in parts),
            "flops": sum(p + 2 * v for p, _, v in parts)}


# ---- the same in plain torch, 64 bits ----

class _Dense:
    """The synchronous rounds on dense vectors: a round is one product of the
    adjacency matrix with the frontier's shares."""

    def __init__(self, off, col):
        self.n, self.deg = len(off) - 1, (off[1:] - off[:-1]).double()
        self.d1 = self.deg.clamp(min=1)
        self.off, self.col = off, col
        self.A = torch.sparse_csr_tensor(off.int(), col,
                                         torch.ones(len(col), dtype=torch.float64, device="cuda"),
                                         size=(self.n, self.n))

    def spread(self, share):
        return torch.mv(self.A, share)

    def unit(self, x):
        r = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        r[x] = 1.0
        return r

    def front(self, r, c):
        return (r >= c * self.deg) & (self.deg > 0)

    def prnibble(self, starts, weights, alpha, eps, rule, beta):
        p = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        r = torch.zeros_like(p)
        r[starts] = weights / weights.sum()
        F = r > 0
        while bool(F.any()):
            if beta < 1.0:
                at = torch.nonzero(F).reshape(-1)
                order = torch.argsort(r[at] / self.d1[at], descending=True, stable=True)
                F = torch.zeros_like(F)
                F[at[order[:max(1, math.ceil(beta * len(at)))]]] = True
            rv = torch.where(F, r, 0.0)
            if rule == "opt":
                p += 2.0 * alpha / (1.0 + alpha) * rv
                r = torch.where(F, 0.0, r)
                share = (1.0 - alpha) / (1.0 + alpha) * rv / self.d1
            else:
                p += alpha * rv
                r = torch.where(F, (1.0 - alpha) * r / 2.0, r)
                share = (1.0 - alpha) * rv / (2.0 * self.d1)
            r = r + self.spread(share)
            F = self.front(r, eps)
        return p

    def nibble(self, x, T, eps):
        p = self.unit(x)
        F = p > 0
        for _ in range(T):
            pf = torch.where(F, p, 0.0)
            q = pf / 2.0 + self.spread(pf / (2.0 * self.d1))
            F = self.front(q, eps)
            if eps == 0.0:
                F &= q > 0
            if not bool(F.any()):
                break
            p = q
        return p

    def hkpr(self, x, t, N, eps):
        psi = [1.0] * (N + 1)
        for k in range(N - 1, -1, -1):
            psi[k] = 1.0 + t / (k + 1) * psi[k + 1]
        r = self.unit(x)
        p = torch.zeros_like(r)
        F = r > 0
        for j in range(N):
            if not bool(F.any()):
                break
            rf = torch.where(F, r, 0.0)
            p += rf
            if j + 1 == N:
                p += self.spread(rf / self.d1)
                break
            r = self.spread(t * rf / ((j + 1) * self.d1))
            F = self.front(r, math.exp(t) * eps / (2.0 * N * psi[j + 1]))
        return p

    def conductance(self, p):
        """The smallest cut / min(vol, 2m - vol) over the prefixes of the
        vertices with p > 0 by p / d, falling."""
        v = torch.nonzero(p > 0).reshape(-1)
        v = v[torch.argsort(p[v] / self.d1[v], descending=True, stable=True)]
        rank = torch.full((self.n,), len(v), dtype=torch.int32, device="cuda")
        rank[v] = torch.arange(len(v), dtype=torch.int32, device="cuda")
        # an edge adds to the boundary at its first end and leaves at its last
        delta = torch.zeros(len(v) + 1, dtype=torch.int64, device="cuda")
        step = 1 << 27
        for a in range(0, len(self.col), step):
            e = torch.arange(a, min(a + step, len(self.col)), device="cuda")
            rs = rank[torch.searchsorted(self.off, e, right=True) - 1]
            rt = rank[self.col[a:a + step].long()]
            up = rs < rt
            one = torch.ones(int(up.sum()), dtype=torch.int64, device="cuda")
            delta.index_add_(0, rs[up], one)
            delta.index_add_(0, rt[up], -one)
        cut = torch.cumsum(delta[:-1], 0)
        vol = torch.cumsum(self.deg[v].long(), 0)
        den = torch.minimum(vol, len(self.col) - vol)
        phi = torch.where(den > 0, cut.double() / den.clamp(min=1), math.inf)
        return float(phi.min()) if len(v) else math.inf


def _philox(walk, draw, key):
    """Words 0 and 1 of Philox4x32-10 (Salmon et al., SC'11), key (low, high),
    counter (walk low, walk high, draw, 0)."""
    mask = 0xFFFFFFFF
    c0, c1, c2, c3 = walk & mask, walk >> 32, torch.full_like(walk, draw), torch.zeros_like(walk)
    k0, k1 = key & mask, key >> 32
    for i in range(10):
        if i:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (b >> 32 & mask) ^ c1 ^ k0, b & mask, (a >> 32 & mask) ^ c3 ^ k1, a & mask
    return c0, c1


def _walks(off, col, x, t, K, walks, key):
    """p of rand-HK-PR: the share of the walks that end at each vertex."""
    cdf, term, total = [], math.exp(-t), 0.0
    for k in range(K):
        total += term
        cdf.append(total)
        term = term * t / (k + 1)
    i = torch.arange(walks, device="cuda")
    w0, w1 = _philox(i, 0, key)
    u = ((w0 << 21) | (w1 >> 11)).double() * 2.0 ** -53
    length = torch.searchsorted(torch.tensor(cdf, dtype=torch.float64, device="cuda"), u, right=True)
    at = torch.full((walks,), x, dtype=torch.int64, device="cuda")
    for s in range(1, K + 1):
        w0, _ = _philox(i, s, key)
        d = off[at + 1] - off[at]
        nxt = col[(off[at] + (w0 * d >> 32)).clamp(max=len(col) - 1)].long()
        at = torch.where(s <= length, nxt, at)
    return torch.bincount(at, minlength=len(off) - 1).double() / walks


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch" and case["B"] * case["n"] > 1 << 25:
        return None  # dense rounds for every seed would take minutes
    off, col, starts, more = _inputs(case, seed)
    D = _Dense(off, col)
    one = np.ones(1)

    def pr(x, w, eps, beta=1.0):
        return D.prnibble(torch.from_numpy(np.asarray(x, np.int64)).cuda(),
                          torch.from_numpy(np.asarray(w, np.float64)).cuda(), case["alpha"], eps,
                          case.get("rule", "opt"), beta)

    def vals(*ps):
        found = np.concatenate([p[p > 0].cpu().numpy() for p in ps])
        return np.concatenate([found, np.zeros(_room(case) - len(found))])

    x = int(starts[0])
    if kind == "batch":
        ps = [pr([v], one, float(more["eps"][i])) for i, v in enumerate(starts)]
        return dict(nnz=None, idx=None, val=vals(*ps),
                    conductance=np.array([D.conductance(p) for p in ps]))
    if kind == "serve":
        ps = [D.hkpr(int(v), float(more["t"][i]), _taylor(float(more["t"][i])), 1e-7)
              if i % 5 == 4 else pr([v], one, float(more["eps"][i]))
              for i, v in enumerate(starts)]
        return [(None, vals(p), D.conductance(p)) for p in ps]
    if kind == "prnibble":
        p = pr([x], one, case["eps"])
    elif kind == "set":
        p = pr(starts, more["weights"], case["eps"], case["beta"])
    elif kind == "nibble":
        p = D.nibble(x, case["T"], case["eps"])
    elif kind == "hkpr":
        p = D.hkpr(x, case["t"], case["N"], case["eps"])
    else:
        p = _walks(off, col, x, case["t"], case["K"], case["walks"], more["rng_seed"])
    cluster = dict(whole=None, conductance=D.conductance(p))
    if case.get("mode", "det") == "det":
        cluster["ids"] = None
    return dict(nnz=None, idx=None, val=vals(p), cluster=cluster)
