"""The work that a user of this library has it do, as cases to time.

Every case goes through the Python entry points of ``paper_1711_00121_gb300``
(``SimRank``, ``MultiSimRank``) on seeded directed power-law graphs (Chung-Lu,
exponent 2.1 or 2.2, the degrees of the repository's own workloads).  The
kinds:

``dense``    a handle with a dense S applies a list of updates, its columns are
             queried, the updates are undone (so that a pass leaves the graph
             as it found it) and the columns are queried again.  The options
             of a case are the handle's: vector and S precision, how many
             updates share an S pass, unit updates, sink blocks or the
             one-shot batch form.
``columns``  a column-mode handle (no dense S) with a few stored updates
             answers a block of column queries.
``grad``     the pair loss and its gradient with respect to the edge weights.
``multi``    many graphs advanced together, then queried and taken back.
``init``     a handle made from an edge list (S by the batch algorithm) and
             a first query.
``anchor``   drift correction of a dense S by sweeps of the batch algorithm.

``exact`` recomputes what a pass returns in FP64 with plain torch operations,
from the definitions: the fixed point of S = C Q S Q^T + (1 - C) I, then per
update the K-truncated series of the rank-one (or rank-2r) Sylvester
equation.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_1711_00121_gb300 as P

DEV = "cuda" if torch.cuda.is_available() else "cpu"


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------
def listed():
    return [
        # one edge arrives, a node is looked up, the edge goes again: the
        # smallest interactive call, default options, columns to the host
        dict(name="one_edge_1k", kind="dense", n=1000, m=8000, C=0.6, K=15, updates=1, query=1,
             host=True),
        # the repository's own update stream: FP32 S, FP64 vectors, the launch
        # shape that the autotuner cached
        dict(name="stream_20k", kind="dense", n=20000, m=200000, C=0.6, K=20, updates=48,
             query=256, vec_fp64=1, tuned=True),
        # a stream at the size of DBLP (13,634 nodes), FP32 vectors, a number of
        # updates that does not fill the last pending group
        dict(name="stream_13k_f32", kind="dense", n=13634, m=93560, C=0.6, K=15, updates=41,
             query=192, tc=2, defer=16),
        # every update visible in S at once: one S pass per update
        dict(name="per_update_16k", kind="dense", n=16001, m=160000, C=0.6, K=20, updates=8,
             query=160, vec_fp64=1, tc=2, defer=0),
        # S in FP64
        dict(name="stream_s64_4k", kind="dense", n=4000, m=31999, C=0.6, K=15, updates=8,
             query=64, s_precision=64),
        # a batch into few sinks as similar-sink blocks, default S passes
        dict(name="sink_blocks_8k", kind="dense", n=8191, m=65000, C=0.6, K=15, updates=48,
             sinks=12, query=128, apply="sink_blocks"),
        # a whole batch as one rank-2r update
        dict(name="one_shot_12k", kind="dense", n=12000, m=180000, C=0.8, K=20, updates=192,
             query=128, apply="one_shot", tc=2, gamma=2.2),
        # a graph whose S is not kept: a block of columns on demand
        dict(name="columns_200k", kind="columns", n=200000, m=2000000, C=0.6, K=15, updates=4,
             query=256),
        # learning edge weights from pairs of scores
        dict(name="grad_5k", kind="grad", n=5000, m=50000, C=0.6, K=15, pairs=600),
        # many small graphs, a few updates each
        dict(name="multi_60", kind="multi", graphs=60, n_lo=500, n_hi=4000, deg=8, C=0.6, K=15,
             updates=6, query=8),
        # a first S from an edge list
        dict(name="init_6k", kind="init", n=6000, m=60000, C=0.6, K=15, query=96),
        # two sweeps of drift correction
        dict(name="anchor_10k", kind="anchor", n=10007, m=100000, C=0.6, K=15, sweeps=2,
             query=128),
    ]


def _span(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm; odd as often as not."""
    v = int(round(lo * (hi / lo) ** rng.random()))
    return max(lo, min(hi, v + rng.randrange(2)))


def draw(rng):
    kind = rng.choice(["one", "stream", "stream", "stream", "per_update", "s64", "sink_blocks",
                       "one_shot", "columns", "grad", "multi", "init", "anchor"])
    c = dict(C=rng.choice([0.6, 0.6, 0.8]), K=rng.randrange(8, 21))
    deg = rng.choice([4, 5, 7, 8, 10, 12])
    if kind == "columns":
        n = _span(rng, 5000, 150000)
        return dict(c, kind="columns", n=n, m=deg * n + rng.randrange(n), updates=rng.randrange(5),
                    query=_span(rng, 3, 256), s_precision=rng.choice([32, 32, 64]),
                    K=rng.randrange(5, 16))
    if kind == "grad":
        n = _span(rng, 500, 5000)
        return dict(c, kind="grad", n=n, m=min(deg, 9) * n, pairs=_span(rng, 30, 500),
                    K=rng.randrange(5, 16))
    if kind == "multi":
        lo = _span(rng, 300, 1500)
        return dict(c, kind="multi", graphs=rng.randrange(8, 50), n_lo=lo, n_hi=lo * 2 + 77,
                    deg=min(deg, 8), updates=rng.randrange(1, 7), query=rng.randrange(1, 9), C=0.6,
                    K=rng.randrange(8, 16))
    if kind == "init":
        n = _span(rng, 400, 6000)
        return dict(c, kind="init", n=n, m=min(deg, 9) * n, query=_span(rng, 1, 96), C=0.6)
    if kind == "anchor":
        n = _span(rng, 1000, 9500)
        return dict(c, kind="anchor", n=n, m=min(deg, 9) * n, sweeps=rng.randrange(1, 3),
                    query=_span(rng, 16, 128), s_precision=rng.choice([32, 32, 64]), C=0.6)
    c["kind"] = "dense"
    if kind == "one":
        n = _span(rng, 300, 4000)
        return dict(c, n=n, m=deg * n, updates=1, query=rng.randrange(1, 5), host=True)
    if kind == "stream":
        n = _span(rng, 1500, 14000)
        return dict(c, n=n, m=min(deg, 10) * n + rng.randrange(99), updates=_span(rng, 9, 64),
                    query=_span(rng, 64, 200), vec_fp64=rng.randrange(2), tc=rng.choice([1, 2, 2]),
                    defer=rng.choice([8, 16, 24]), C=0.6)
    if kind == "per_update":
        n = _span(rng, 2000, 12000)
        return dict(c, n=n, m=min(deg, 10) * n, updates=_span(rng, 2, 8), query=_span(rng, 64, 160),
                    vec_fp64=rng.randrange(2), tc=rng.choice([0, 2]), defer=0, C=0.6)
    if kind == "s64":
        n = _span(rng, 500, 4000)
        return dict(c, n=n, m=deg * n, updates=_span(rng, 2, 8), query=_span(rng, 16, 64),
                    s_precision=64, C=0.6)
    if kind == "sink_blocks":
        n = _span(rng, 1000, 8000)
        return dict(c, n=n, m=deg * n, updates=_span(rng, 16, 64), sinks=_span(rng, 3, 12),
                    query=_span(rng, 32, 128), apply="sink_blocks", tc=rng.choice([0, 0, 2]), C=0.6)
    n = _span(rng, 1000, 10000)
    return dict(c, n=n, m=deg * n, updates=_span(rng, 16, 192), query=_span(rng, 32, 128),
                apply="one_shot", tc=rng.choice([1, 2, 2]))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _graph(n, m, gamma, rng):
    """A directed Chung-Lu graph: m distinct edges, no self-loop, power-law
    in- and out-weights (independent permutations).  Keys src * n + dst."""
    w = (np.arange(n) + 1.0) ** (-1.0 / (gamma - 1.0))
    out_cdf = np.cumsum(w[rng.permutation(n)])
    in_cdf = np.cumsum(w[rng.permutation(n)])
    keys = np.empty(0, np.int64)
    while keys.size < m:
        k = int(1.4 * (m - keys.size)) + 64
        s = np.searchsorted(out_cdf, rng.random(k) * out_cdf[-1], side="right").clip(0, n - 1)
        d = np.searchsorted(in_cdf, rng.random(k) * in_cdf[-1], side="right").clip(0, n - 1)
        keys = np.unique(np.concatenate([keys, (s * np.int64(n) + d)[s != d]]))
    return rng.permutation(keys)[:m]


def _split(keys, n):
    return (keys // n).astype(np.int32), (keys % n).astype(np.int32)


def _updates(n, keys, count, rng, sinks=0):
    """count updates of distinct edges in random order: about 80% insertions
    (endpoints drawn by degree + 1; into `sinks` chosen nodes when set), the
    rest deletions of edges of the graph."""
    src, dst = keys // n, keys % n
    out_cdf = np.cumsum(np.bincount(src, minlength=n) + 1.0)
    in_cdf = np.cumsum(np.bincount(dst, minlength=n) + 1.0)
    n_del = 0 if count == 1 else int(round(0.2 * count))
    dele = rng.choice(keys, size=n_del, replace=False)
    sinkset = None
    if sinks:
        sinkset = np.unique(np.searchsorted(in_cdf, rng.random(4 * sinks) * in_cdf[-1],
                                            side="right").clip(0, n - 1))
        sinkset = rng.permutation(sinkset)[:sinks]
    ins = np.empty(0, np.int64)
    while ins.size < count - n_del:
        k = 4 * count + 64
        s = np.searchsorted(out_cdf, rng.random(k) * out_cdf[-1], side="right").clip(0, n - 1)
        if sinks:
            d = sinkset[rng.integers(0, sinkset.size, k)]
        else:
            d = np.searchsorted(in_cdf, rng.random(k) * in_cdf[-1], side="right").clip(0, n - 1)
        c = (s * np.int64(n) + d)[s != d]
        c = c[~np.isin(c, keys)]
        ins = rng.permutation(np.unique(np.concatenate([ins, c])))
    ins = ins[:count - n_del]
    k = np.concatenate([ins, dele])
    op = np.concatenate([np.ones(ins.size, np.int64), -np.ones(n_del, np.int64)])
    o = rng.permutation(count)
    k, op = k[o], op[o]
    return np.stack([k // n, k % n, op], 1).astype(np.int32)


def _undo(ups):
    back = ups[::-1].copy()
    back[:, 2] *= -1
    return back


def _inputs(case, seed):
    """Everything a pass reads, made from the seed alone."""
    rng = np.random.default_rng([int(seed), 17])
    if case["kind"] == "multi":
        graphs, ups, cols = [], [], []
        for g in range(case["graphs"]):
            # sizes spread evenly over the range, 1 to `updates` updates each
            n = case["n_lo"] + (case["n_hi"] - case["n_lo"]) * g // max(1, case["graphs"] - 1)
            keys = _graph(n, case["deg"] * n, 2.1, rng)
            graphs.append((n, *_split(keys, n)))
            ups.append(_updates(n, keys, 1 + g % case["updates"], rng))
            cols.append(rng.choice(n, case["query"], replace=False).astype(np.int32))
        return dict(graphs=graphs, ups=ups, cols=cols)
    n, m = case["n"], case["m"]
    keys = _graph(n, m, case.get("gamma", 2.1), rng)
    src, dst = _split(keys, n)
    x = dict(n=n, src=src, dst=dst)
    if case["kind"] == "grad":
        x["w"] = (1.0 - 0.9 * rng.random(m)).astype(np.float32)
        a = rng.integers(0, n, case["pairs"])
        b = rng.integers(0, n - 1, case["pairs"])
        x["a"], x["b"] = a.astype(np.int32), (b + (b >= a)).astype(np.int32)
        x["t"] = rng.uniform(0.0, 0.3, case["pairs"])
        return x
    x["cols"] = rng.choice(n, case["query"], replace=False).astype(np.int32)
    if case.get("updates"):
        x["ups"] = _updates(n, keys, case["updates"], rng, case.get("sinks", 0))
    return x


_APPLY = {"unit": P.APPLY_UNIT, "sink_blocks": P.APPLY_SINK_BLOCKS, "one_shot": P.APPLY_ONE_SHOT}
_INIT_TOL = 1e-9  # of the S that a prepared handle starts from (FP32 S)


def _config(case):
    kw = dict(C=case["C"], K=case["K"], s_precision=case.get("s_precision", 32))
    for k in ("vec_fp64", "tc", "defer", "tuned"):
        if k in case:
            kw[k] = case[k]
    if "apply" in case:
        kw["apply"] = _APPLY[case["apply"]]
    return kw


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "multi":
        h = P.MultiSimRank(x["graphs"], C=case["C"], K=case["K"], s_precision=32, init_tol=1e-9, tc=1)
        packed = []
        for ups in (x["ups"], [_undo(u) for u in x["ups"]]):
            arrs = [P.updates_array(u) for u in ups]
            off = np.zeros(len(arrs) + 1, np.int64)
            off[1:] = np.cumsum([a.size for a in arrs])
            packed.append((np.ascontiguousarray(np.concatenate(arrs)), off))
        return dict(kind=kind, h=h, packed=packed, cols=x["cols"])
    if kind == "init":
        return dict(kind=kind, x=x, kw=_config(case))
    if kind == "grad":
        h = P.SimRank(x["n"], x["src"], x["dst"], weight=x["w"], C=case["C"], K=case["K"],
                      s_precision=64, mode=P.MODE_COLUMN, stream=_stream())
        return dict(kind=kind, h=h, x=x, m=case["m"])
    kw = _config(case)
    f64 = kw["s_precision"] == 64
    if kind == "columns":
        h = P.SimRank(x["n"], x["src"], x["dst"], mode=P.MODE_COLUMN, stream=_stream(), **kw)
        if "ups" in x:
            h.apply_updates(x["ups"])
    else:
        h = P.SimRank(x["n"], x["src"], x["dst"], init_tol=1e-13 if f64 else _INIT_TOL,
                      stream=_stream(), **kw)
    st = dict(kind=kind, h=h, cols=x["cols"], host=case.get("host", False),
              sweeps=case.get("sweeps"))
    dt = torch.float64 if f64 else torch.float32
    st["out"] = [torch.empty((case["query"], x["n"]), dtype=dt, device="cuda") for _ in range(2)]
    if kind == "dense":
        st["ups"] = P.updates_array(x["ups"])
        st["back"] = P.updates_array(_undo(x["ups"]))
    return st


def run(st):
    kind = st["kind"]
    if kind == "init":
        x = st["x"]
        h = P.SimRank(x["n"], x["src"], x["dst"], **st["kw"])
        out = h.columns(x["cols"], fp64=False)
        h.close()
        return out
    h = st["h"]
    if kind == "grad":
        x = st["x"]
        loss, g = h.grad(x["a"], x["b"], x["t"], st["m"])
        return dict(loss=loss, grad=g)
    if kind == "multi":
        h.apply_packed(*st["packed"][0])
        out = [h.columns(g, c, fp64=False) for g, c in enumerate(st["cols"])]
        h.apply_packed(*st["packed"][1])
        return out
    if kind == "columns":
        h.columns_device(st["cols"], st["out"][0])
        return st["out"][0]
    if kind == "anchor":
        h.reanchor(st["sweeps"])
        h.columns_device(st["cols"], st["out"][0])
        return st["out"][0]
    if st["host"]:
        h.apply_updates(st["ups"])
        a = h.columns(st["cols"], fp64=False)
        h.apply_updates(st["back"])
        return [a, h.columns(st["cols"], fp64=False)]
    h.apply_updates(st["ups"])
    h.columns_device(st["cols"], st["out"][0])
    h.apply_updates(st["back"])
    h.columns_device(st["cols"], st["out"][1])
    return st["out"]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    K1 = case["K"] + 1
    kind = case["kind"]
    if kind == "multi":
        n = 0.5 * (case["n_lo"] + case["n_hi"])
        sq = (n * n + (case["n_hi"] - case["n_lo"]) ** 2 / 12.0) * case["graphs"]
        ups = 0.5 * (case["updates"] + 1)
        m = case["deg"] * n * case["graphs"]
        # both calls read and write the upper triangle of every S
        return dict(bytes=2 * sq * 4.0 + 2 * 4 * m + case["query"] * n * case["graphs"] * 4.0,
                    flops=2 * ups * (2.0 * K1 * sq + 4.0 * K1 * m))
    n, m = case["n"], case["m"]
    eb = case.get("s_precision", 32) / 8.0
    if kind == "grad":
        ends = min(n, 2 * case["pairs"])
        return dict(bytes=24.0 * m + 16.0 * case["pairs"],
                    flops=2.0 * m * case["K"] * (2 * min(n, case["pairs"]) + 4 * ends))
    if kind == "columns":
        q = case["query"]
        return dict(bytes=8.0 * m + q * n * eb + case["updates"] * 2.0 * K1 * n * eb,
                    flops=4.0 * case["K"] * m * q + 4.0 * K1 * case["updates"] * n * q)
    if kind == "init":
        # sweeps until the change, which shrinks by C each time, is below 1e-13
        sweeps = np.ceil(np.log(1e-13) / np.log(case["C"]))
        return dict(bytes=8.0 * m + n * n * eb + case["query"] * n * 4.0,
                    flops=float(sweeps * 4.0 * m * n))
    q = case["query"] * n * eb
    if kind == "anchor":
        return dict(bytes=2.0 * n * n * eb + 4.0 * m + q, flops=case["sweeps"] * 4.0 * m * n)
    # dense: each of the two calls reads and writes the upper triangle of S
    blocks = min(case.get("sinks", 1 << 30), case["updates"])
    if case.get("apply") == "sink_blocks":
        blocks = 1.3 * blocks
    return dict(bytes=2 * (n * n * eb + 4.0 * m + q),
                flops=2 * blocks * (2.0 * K1 * n * n + 4.0 * K1 * m))


# --------------------------------------------------------------------------
# the same in FP64, from the definitions
# --------------------------------------------------------------------------
class _Graph:
    """A changing directed graph and products with its Q (Q[a][b] =
    1 / in-degree(a) for an edge b -> a) in FP64."""

    def __init__(self, n, src, dst, w=None):
        self.n = n
        self.src = torch.as_tensor(np.asarray(src, np.int64), device=DEV)
        self.dst = torch.as_tensor(np.asarray(dst, np.int64), device=DEV)
        self.w = None if w is None else torch.as_tensor(w.astype(np.float64), device=DEV)
        self._deg()

    def _deg(self):
        w = torch.ones(self.src.numel(), dtype=torch.float64, device=DEV) if self.w is None else self.w
        self.deg = torch.zeros(self.n, dtype=torch.float64, device=DEV).index_add_(0, self.dst, w)
        self.val = w / self.deg[self.dst]

    def edge(self, i, j, op):
        if op > 0:
            self.src = torch.cat([self.src, torch.tensor([i], device=DEV)])
            self.dst = torch.cat([self.dst, torch.tensor([j], device=DEV)])
        else:
            keep = ~((self.src == i) & (self.dst == j))
            self.src, self.dst = self.src[keep], self.dst[keep]
        self._deg()

    def _mm(self, x, to, fr):
        y = torch.zeros_like(x)
        step = max(1, (1 << 29) // max(1, self.src.numel()))
        for c in range(0, x.shape[1], step):
            y[:, c:c + step].index_add_(0, to, x[:, c:c + step][fr] * self.val[:, None])
        return y

    def q(self, x):
        return self._mm(x, self.dst, self.src)

    def qt(self, x):
        return self._mm(x, self.src, self.dst)

    def csr(self):
        o = torch.argsort(self.dst)
        crow = torch.zeros(self.n + 1, dtype=torch.int64, device=DEV)
        crow[1:] = torch.cumsum(torch.bincount(self.dst, minlength=self.n), 0)
        return torch.sparse_csr_tensor(crow, self.src[o], self.val[o], (self.n, self.n))


def _sweep(q, S, C):
    T = torch.mm(q, torch.mm(q, S).T.contiguous()).mul_(C)
    T.diagonal().add_(1.0 - C)
    return T


def _fixed_point(g, C, tol=1e-14):
    q = g.csr()
    S = torch.eye(g.n, dtype=torch.float64, device=DEV).mul_(1.0 - C)
    for _ in range(int(np.ceil(np.log(tol) / np.log(C))) + 2):
        S = _sweep(q, S, C)
    return S


class _Dense:
    """S of a graph under updates: S0 plus accumulated X H^T + H X^T."""

    def __init__(self, n, src, dst, C, K):
        self.g, self.C, self.K = _Graph(n, src, dst), C, K
        self.S0 = _fixed_point(self.g, C)
        self.X, self.H = [], []

    def rows(self, ids):
        """S[ids, :] as columns (n x len(ids))."""
        r = self.S0[ids].T.clone()
        for X, H in zip(self.X, self.H):
            r += X @ H[ids].T + H @ X[ids].T
        return r

    def _series(self, xi, eta):
        """Adds sum_k C^k Q^k (xi eta^T + eta xi^T) Q^kT."""
        r = xi.shape[1]
        v = torch.cat([xi, eta], 1)
        X, H = [v[:, :r]], [v[:, r:]]
        for _ in range(self.K):
            v = self.g.q(v)
            v[:, :r] *= self.C
            X.append(v[:, :r].clone())
            H.append(v[:, r:].clone())
        self.X.append(torch.cat(X, 1))
        self.H.append(torch.cat(H, 1))

    def block(self, I, j, op):
        """Sources I into (op = 1) or out of (op = -1) the sink j."""
        sI = self.rows(I).sum(1, keepdim=True)
        sJ = self.rows([j])
        self.apply(I, j, op, sI, sJ)

    def apply(self, I, j, op, sI, sJ):
        g, C, n = self.g, self.C, self.g.n
        d = float(g.deg[j])
        dn = d + op * len(I)
        if d == 0:
            a, b = 0.0, 1.0 / dn
        elif dn == 0:
            a, b = 0.0, -1.0 / d
        else:
            a, b = d / dn - 1.0, op / dn
        ej = torch.zeros(n, 1, dtype=torch.float64, device=DEV)
        ej[j] = 1.0
        y = g.q(sI)
        lam = (a * a * (sJ[j] - (1 - C)) / C + 2 * a * b * y[j] + b * b * sI[I].sum())
        eta = a * (sJ - (1 - C) * ej) / C + b * y + 0.5 * lam * ej
        for i in I:
            g.edge(i, j, op)
        self._series(C * ej, eta)

    def unit(self, ups):
        for i, j, op in ups.tolist():
            self.block([i], j, op)

    def sink_blocks(self, ups):
        """Deletions by ascending sink, then insertions by ascending sink."""
        for op in (-1, 1):
            sel = ups[ups[:, 2] == op]
            for j in np.unique(sel[:, 1]).tolist():
                self.block(sorted(sel[sel[:, 1] == j, 0].tolist()), j, op)

    def one_shot(self, ups):
        g, C, n = self.g, self.C, self.g.n
        sinks = np.unique(ups[:, 1]).tolist()
        r = len(sinks)
        av, bv, src = [], [], []
        for j in sinks:
            u = ups[ups[:, 1] == j]
            d = float(g.deg[j])
            dn = d + int(u[:, 2].sum())
            if d == 0:
                a, b = 0.0, 1.0 / dn
            elif dn == 0:
                a, b = -1.0, 0.0
            else:
                a, b = d / dn - 1.0, 1.0 / dn
            av.append(a)
            bv.append(b)
            src.append(u[:, [0, 2]].tolist())
        av = torch.tensor(av, dtype=torch.float64, device=DEV)
        bv = torch.tensor(bv, dtype=torch.float64, device=DEV)
        U = torch.zeros(n, r, dtype=torch.float64, device=DEV)
        U[sinks, torch.arange(r, device=DEV)] = 1.0
        D = torch.zeros(n, r, dtype=torch.float64, device=DEV)  # signed sources
        for t, u in enumerate(src):
            for i, op in u:
                D[i, t] += op
        SJ = self.rows(sinks)
        ids = sorted({i for u in src for i, _ in u})
        Z = self.rows(ids) @ D[ids]
        Y = g.q(Z)
        qsq = (SJ - (1 - C) * U) / C
        lam = (av[:, None] * av[None, :] * qsq[sinks]
               + av[:, None] * bv[None, :] * Y[sinks] + bv[:, None] * av[None, :] * Y[sinks].T
               + bv[:, None] * bv[None, :] * (D.T @ Z))
        W = qsq * av + Y * bv + U @ lam / 2
        for i, j, op in ups.tolist():
            g.edge(i, j, op)
        self._series(C * U, W)


def _partial(g, e, C, K):
    """(1-C) sum_{k<=K} C^k Q^k (Q^T)^k e."""
    xs = [e]
    for _ in range(K):
        xs.append(g.qt(xs[-1]))
    y = xs[K]
    for t in range(1, K + 1):
        y = xs[K - t] + C * g.q(y)
    return (1.0 - C) * y


class _Columns(_Dense):
    """The same without a dense S: old columns by the truncated series."""

    def __init__(self, n, src, dst, C, K):
        self.g, self.C, self.K = _Graph(n, src, dst), C, K
        self.g0 = _Graph(n, src, dst)
        self.X, self.H = [], []

    def _unit_cols(self, ids):
        e = torch.zeros(self.g.n, len(ids), dtype=torch.float64, device=DEV)
        e[torch.as_tensor(ids, dtype=torch.int64, device=DEV), torch.arange(len(ids), device=DEV)] = 1.0
        return e

    def block(self, I, j, op):
        s = _partial(self.g, self._unit_cols(list(I) + [j]), self.C, self.K)
        self.apply(I, j, op, s[:, :-1].sum(1, keepdim=True), s[:, -1:])

    def rows(self, ids):
        r = _partial(self.g0, self._unit_cols(ids), self.C, self.K)
        for X, H in zip(self.X, self.H):
            r += X @ H[ids].T + H @ X[ids].T
        return r


def _grad(x, C, K):
    n = x["n"]
    g = _Graph(n, x["src"], x["dst"], x["w"])
    a = torch.as_tensor(x["a"].astype(np.int64), device=DEV)
    b = torch.as_tensor(x["b"].astype(np.int64), device=DEV)
    t = torch.as_tensor(x["t"], device=DEV)
    ends, inv = torch.unique(torch.cat([a, b]), return_inverse=True)
    ia, ib = inv[:a.numel()], inv[a.numel():]
    E = torch.zeros(n, ends.numel(), dtype=torch.float64, device=DEV)
    E[ends, torch.arange(ends.numel(), device=DEV)] = 1.0
    S = _partial(g, E, C, K)
    r = S[a, ib] - t
    loss = float((r * r).sum())
    # G = dL/dS + its transpose, in the columns of the endpoints
    psi = torch.zeros_like(E)
    psi.index_put_((b, ia), 2 * r, accumulate=True)
    psi.index_put_((a, ib), 2 * r, accumulate=True)
    F, V = [E], [psi]
    for _ in range(K):
        F.append(g.qt(F[-1]))
        V.append(g.qt(V[-1]))
    dq = torch.zeros_like(g.val)
    y = torch.zeros_like(E)
    for k in range(K - 1, -1, -1):
        y = C ** (k + 1) * V[k + 1] + g.q(y)
        dq += (1.0 - C) * (F[k][g.dst] * y[g.src]).sum(1)
    # through Q[a][b] = w / (sum of row a's weights)
    mean = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, g.dst, dq * g.val)
    return dict(loss=loss, grad=((dq - mean[g.dst]) / g.deg[g.dst]).cpu().numpy())


def exact(case, seed):
    x = _inputs(case, seed)
    kind, C, K = case["kind"], case["C"], case["K"]
    if kind == "grad":
        return _grad(x, C, K)
    if kind == "multi":
        out = []
        for (n, s, d), ups, cols in zip(x["graphs"], x["ups"], x["cols"]):
            S = _Dense(n, s, d, C, K)
            S.unit(ups)
            out.append(S.rows(cols.tolist()).cpu().numpy())
        return out
    n, cols = x["n"], x["cols"].tolist()
    if kind == "init":
        return _fixed_point(_Graph(n, x["src"], x["dst"]), C)[:, cols].cpu().numpy()
    if kind == "anchor":
        return _fixed_point(_Graph(n, x["src"], x["dst"]), C)[cols].cpu()
    if kind == "columns":
        S = _Columns(n, x["src"], x["dst"], C, K)
        if "ups" in x:
            S.unit(x["ups"])
        return S.rows(cols).T.contiguous().cpu()
    S = _Dense(n, x["src"], x["dst"], C, K)
    apply = getattr(S, case.get("apply", "unit"))
    out = []
    for ups in (x["ups"], _undo(x["ups"])):
        apply(ups)
        r = S.rows(cols)
        out.append(r.cpu().numpy() if case.get("host") else r.T.contiguous().cpu())
    return out
