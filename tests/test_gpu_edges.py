"""Kernels at the sizes where their splits end: row chunks, tiles, remainders.
Small graphs against the oracle, through the C ABI."""
import numpy as np
import pytest

from oracle import simrank_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1711_00121_gb300 as P

    return P


def degrees_graph(n, degs, seed, reverse=False):
    """Node t < len(degs) has degs[t] in-neighbours (out-neighbours with
    reverse), the others a few each."""
    rng = np.random.default_rng(seed)
    edges = set()
    for t, k in enumerate(list(degs) + [3] * (n - len(degs))):
        for x in rng.choice(np.setdiff1d(np.arange(n), [t]), size=k, replace=False).tolist():
            edges.add((t, x) if reverse else (x, t))
    e = np.array(sorted(edges), np.int32)
    return e[:, 0].copy(), e[:, 1].copy()


@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("prec,width", [(64, 5), (64, 130), (32, 6), (32, 129)])
def test_column_blocks_at_chunk_edges(P, prec, width, reverse):
    """Column queries over rows of 0, 1, 31..33, 64, 65 and 200 nonzeros (row
    chunks hold 32) in both directions, at widths that need padded columns and
    more than one column group.  The values are at most 1 and each is a sum of
    K + 1 = 6 terms: 1e-12 in FP64, 1e-6 in FP32."""
    n, C, K = 300, 0.6, 5
    s, d = degrees_graph(n, [0, 1, 31, 32, 33, 64, 65, 200, 0], 3, reverse)
    sr = P.SimRank(n, s, d, C=C, K=K, s_precision=prec, mode=P.MODE_COLUMN)
    cols = np.random.default_rng(width).choice(n, size=width, replace=False).astype(np.int32)
    got = sr.columns(cols)
    want = O.partial_sim_block(O.transition_matrix(n, s, d, sparse=True), cols, K, C)
    assert np.max(np.abs(got - want)) < (1e-12 if prec == 64 else 1e-6)


def sweeps(S, Q, C, k):
    for _ in range(k):
        S = C * (Q @ (Q @ S).T).T + (1.0 - C) * np.eye(S.shape[0])
    return S


@pytest.mark.parametrize("C", [0.6, 0.25, 0.95])
@pytest.mark.parametrize("n,degs", [(300, [0, 1, 2, 95, 96, 97, 100, 131, 257, 0]), (1, []), (65, [64, 1])])
def test_fixed_point_sweeps_at_row_edges(P, n, degs, C):
    """The first S of an FP64 handle (fixed-point sweeps: rows of up to 96
    nonzeros by one warp, longer ones by the CTA) and one sweep more, against
    the oracle's fixed point: both stop within C / (1 - C) 1e-13 of it."""
    s, d = degrees_graph(n, degs, 5) if n > 1 else (np.zeros(0, np.int32), np.zeros(0, np.int32))
    sr = P.SimRank(n, s, d, C=C, K=3, s_precision=64, init_max_sweeps=2000)
    want = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-15)
    tol = 1e-13 * C / (1.0 - C) + 1e-14
    assert np.max(np.abs(sr.dense() - want)) < tol
    sr.reanchor(1)
    assert np.max(np.abs(sr.dense() - want)) < tol


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("form", ["symmetric", "rounded", "asymmetric", "large", "negative"])
def test_sweeps_from_any_s0(P, form, prec):
    """Sweeps from a caller's S0: symmetric entries below 1.875 in magnitude
    (also when symmetric only up to rounding) run in fixed point, others (an
    asymmetric S0, one entry of 40) in FP64; all give the sweeps of the
    symmetrised S0.  Entries are at most 40 and a sweep contracts: 1e-13 x 40
    in FP64, 1e-6 x 40 stored in FP32."""
    n, C = 200, 0.6
    s, d = degrees_graph(n, [0, 1, 97, 130, 33], 7)
    rng = np.random.default_rng(8)
    S0 = rng.uniform(-0.5 if form == "negative" else 0.0, 1.0, (n, n))
    if form == "asymmetric":
        S0[3, 7] += 0.25
    else:
        S0 = 0.5 * (S0 + S0.T)
    if form == "large":
        S0[5, 5] = 40.0
    if form == "rounded":
        S0[9, 4] = np.nextafter(S0[9, 4], 2.0)
    dt = np.float64 if prec == 64 else np.float32
    S0 = S0.astype(dt)
    Q = O.transition_matrix(n, s, d)
    sr = P.SimRank(n, s, d, S0=S0, C=C, K=3, s_precision=prec, upper_only=0)
    first = sr.reanchor(1)
    got = sr.dense()
    W = S0.astype(np.float64)
    want = sweeps(W, Q, C, 1)
    tol = (1e-13 if prec == 64 else 1e-6) * 40
    assert np.max(np.abs(got - 0.5 * (want + want.T))) < tol
    assert abs(first - np.max(np.abs(want - W))) < tol
    sr.reanchor(3)
    want = sweeps(0.5 * (W + W.T), Q, C, 4)
    assert np.max(np.abs(sr.dense() - want)) < tol


@pytest.mark.parametrize("prec,kw", [(64, {}), (64, {"prep_ctas": 5}), (32, {"vec_fp64": 1}),
                                     (32, {"tc": 1, "defer": 3, "prep_ctas": 7})])
@pytest.mark.parametrize("scale", [1.0, 1e-20, 1e20])
def test_recurrence_at_warp_and_cta_edges(P, prec, kw, scale):
    """Updates on a graph whose rows end at the splits of the recurrence: 32 and
    64 nonzeros (warps), 256, 512 and 1,024 (CTAs, one or two nonzeros per
    thread), hubs over several CTAs, with fewer CTAs too (longer ranges), and
    an S0 of other magnitudes (the fixed-point exponents).  One update changes
    S by at most its truncated series: 1e-10 of the largest entry in FP64 and
    1e-6 in FP32, as in the parity tests."""
    n, C, K = 1300, 0.6, 7
    degs = [0, 1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025]
    s, d = degrees_graph(n, degs, 11)
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-14) * scale
    edges = set(zip(s.tolist(), d.tolist()))
    sr = P.SimRank(n, s, d, S0=S0, C=C, K=K, s_precision=prec, **kw)
    want = S0.astype(np.float64 if prec == 64 else np.float32).astype(np.float64)
    ups = []
    for j, op in ((19, 1), (0, 1), (3, -1), (1, -1), (700, 1)):
        cand = [x for x in range(n) if x != j and ((x, j) in edges) == (op < 0)]
        ups.append((cand[len(cand) // 2], j, op))
    want, _ = O.sequential_unit_updates(n, s, d, want, ups, C, K)
    sr.apply_updates(ups)
    err = np.max(np.abs(sr.dense() - want)) / max(1.0, np.max(np.abs(want)))
    assert err < (1e-10 if prec == 64 else 1e-6)


@pytest.mark.parametrize("prec,tc", [(64, 0), (32, 0), (32, 1), (32, 2)])
@pytest.mark.parametrize("sinks", [1, 3, 33, 70])
def test_one_shot_at_chunk_and_column_edges(P, prec, tc, sinks):
    """A batch as one rank-2r update on rows of 31..33, 64, 65 and 200 nonzeros
    (row chunks hold 32), with 2 r columns inside one column group of 128 and
    over it: one insertion into every sink, one deletion.  1e-10 (FP64) and
    1e-6 (FP32), as in the one-shot parity tests."""
    n, C, K = 300, 0.6, 6
    s, d = degrees_graph(n, [0, 1, 31, 32, 33, 64, 65, 200], 13)
    edges = set(zip(s.tolist(), d.tolist()))
    ups = [(next(x for x in range(n) if x != j and (x, j) not in edges), j, 1) for j in range(sinks)]
    ups.append((sorted(e for e in edges if e[1] == 7)[0][0], 7, -1))
    ups = [u for u in ups if not (u[1] == 7 and u[2] == 1)]
    new = (edges | {(i, j) for i, j, op in ups if op > 0}) - {(i, j) for i, j, op in ups if op < 0}
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-15)
    sr = P.SimRank(n, s, d, C=C, K=K, s_precision=prec, tc=tc, apply=P.APPLY_ONE_SHOT)
    sr.apply_updates(ups)
    ns, nd = (np.array(v, np.int64) for v in zip(*sorted(new)))
    want = O.one_shot_batch(n, s, d, ns, nd, S0, C, K)
    assert np.max(np.abs(sr.dense() - want)) < (1e-10 if prec == 64 else 1e-6)


@pytest.mark.parametrize("prec", [64, 32])
def test_many_graphs_at_run_edges(P, prec):
    """Many-graph rounds whose runs cut rows at their edges: graphs of one node
    and of a few edges (most threads without a run), rows of 31..33 nonzeros (the
    two loading forms), rows longer than a thread's, a warp's and several
    warps' runs, and a graph too large for the index form.  1e-10 (FP64) and
    1e-6 (FP32), as in the many-graph parity tests."""
    C, K = 0.6, 6
    shapes = [(1, []), (3, [1]), (200, [0, 1, 31, 32, 33, 64, 65, 130]),
              (1100, [1023, 700, 333, 5, 0, 96]), (4700 if prec == 64 else 6500, [900, 40])]
    graphs, ups = [], []
    for t, (n, degs) in enumerate(shapes):
        if n == 1:
            s = d = np.zeros(0, np.int32)
        elif n == 3:
            s, d = np.array([1], np.int32), np.array([0], np.int32)
        else:
            s, d = degrees_graph(n, degs, 17 + t)
        edges = set(zip(s.tolist(), d.tolist()))
        u = []
        for j in range(min(n, 3) if n > 1 else 0):
            i = next((x for x in range(n - 1, -1, -1) if x != j and (x, j) not in edges), None)
            if i is not None:
                u.append((i, j, 1))
        if n > 3:
            u.append((sorted(e for e in edges if e[1] == 2)[0][0], 2, -1))
        graphs.append((n, s, d))
        ups.append(np.array(u, np.int32).reshape(-1, 3))
    mh = P.MultiSimRank(graphs, C=C, K=K, s_precision=prec)
    mh.apply_updates(ups)
    mh.sync()
    for g, (n, s, d) in enumerate(graphs):
        cols = np.unique(np.r_[0, n // 2, n - 1, [u for u in ups[g][:, 1].tolist()]]).astype(np.int32)
        got = mh.columns(g, cols)
        if n > 2000:
            sr = P.SimRank(n, s, d, C=C, K=K, s_precision=64)
            sr.apply_updates(ups[g])
            want = sr.columns(cols)
        else:
            S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-14)
            want = O.sequential_unit_updates(n, s, d, S0, ups[g].tolist(), C, K)[0][:, cols]
        assert np.max(np.abs(got - want)) < (1e-10 if prec == 64 else 1e-6), g


@pytest.mark.parametrize("prec,K,n,kw", [(64, 2, 2, {}), (64, 14, 2, {}), (64, 15, 700, {}),
                                         (64, 16, 641, {"aff": 0}), (64, 32, 640, {}),
                                         (32, 11, 5000, {}), (32, 15, 5120, {"aff": 0})])
@pytest.mark.parametrize("form", ["plain", "huge", "tiny", "inf"])
def test_digit_pass_at_term_and_tile_edges(P, prec, K, n, kw, form):
    """The S pass by exact digits: 3, 15, 16, 17 and 33 terms (16 a pass), node
    counts at and off the tiles of 128, all pairs or the affected ones, entries
    of S0 of other magnitudes, and the direct sum at an infinite entry (inf and
    NaN where the pass of a mirrored S has them).  Relative to the largest
    entry, an update's terms and S are rounded to 2^-53 (FP32: 2^-24) some
    2 (K + 1) + 1 times, as in the product of the oracle: 4 updates, K <= 32,
    stay below 4 * 67 * 2^-52 < 1e-13 (FP32: 4 * 67 * 2^-24 < 2e-5)."""
    C = 0.6
    s, d = degrees_graph(n, [0, 1, 5, 64, 65][:n], 17)
    edges = set(zip(s.tolist(), d.tolist()))
    if n < 1000:
        S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-14)
    else:
        S0 = np.random.default_rng(5).random((n, n))
        S0 = 0.5 * (S0 + S0.T)
    S0 *= {"huge": 1e12, "tiny": 1e-12}.get(form, 1.0)
    if form == "inf":
        S0[0, 0] = np.inf
    ups = []
    for j, op in ((0, 1), (4, 1), (3, -1), (n // 2, 1)):
        j %= n
        cand = [x for x in range(n) if x != j and ((x, j) in edges) == (op < 0)]
        if cand and (cand[len(cand) // 2], j) not in [u[:2] for u in ups]:
            ups.append((cand[len(cand) // 2], j, op))
    sr = P.SimRank(n, s, d, S0=S0, C=C, K=K, s_precision=prec, upper_only=1, **kw)
    sr.apply_updates(ups)
    got = sr.dense()
    if form == "inf":
        old = P.SimRank(n, s, d, S0=S0, C=C, K=K, s_precision=prec, upper_only=0, **kw)
        old.apply_updates(ups)
        want = old.dense()
        np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
        np.testing.assert_array_equal(np.isinf(got), np.isinf(want))
        ok = np.isfinite(want)
    else:
        want = S0.astype(np.float64 if prec == 64 else np.float32).astype(np.float64)
        want, _ = O.sequential_unit_updates(n, s, d, want, ups, C, K)
        ok = np.ones_like(want, bool)
    if ok.any():
        err = np.max(np.abs(got[ok] - want[ok])) / max(1e-12, np.max(np.abs(want[ok])))
        assert err < (1e-13 if prec == 64 else 2e-5)


@pytest.mark.parametrize("prec", [64, 32])
def test_recurrence_with_a_hub_over_many_ctas(P, prec):
    """A row with a quarter of all nonzeros: its sums come in some fifty parts
    (of at most 60), beside rows without nonzeros, whose sums are complete from the
    start.  1e-10 (FP64) and 1e-6 (FP32), as in the parity tests."""
    n, C, K = 9000, 0.6, 3
    s, d = degrees_graph(n, [0, 8500, 0], 23)
    edges = set(zip(s.tolist(), d.tolist()))
    S0 = np.eye(n) * 0.5
    S0[:200, :200] += 0.25
    ups = [(next(x for x in range(2, n) if (x, 1) not in edges), 1, 1), (5, 0, 1),
           (next(x for x, y in sorted(edges) if y == 1), 1, -1), (1, 2, 1)]
    sr = P.SimRank(n, s, d, S0=S0, C=C, K=K, s_precision=prec)
    sr.apply_updates(ups)
    want, _ = O.sequential_unit_updates(n, s, d, S0, ups, C, K)
    assert np.max(np.abs(sr.dense() - want)) < (1e-10 if prec == 64 else 1e-6)


@pytest.mark.parametrize("prec,n", [(64, 700), (32, 5000)])
def test_digit_pass_timeout(P, prec, n):
    """A bound of one poll runs out in the digit pass (the work before it is the
    per-step path, whose kernels have no waits): status 7 from sync, and the device
    stays usable."""
    s, d = degrees_graph(n, [0, 5], 29)
    S0 = np.eye(n) * 0.5
    ups = [(x, 0, 1) for x in range(2, 10)]
    h = P.SimRank(n, s, d, S0=S0, C=0.6, K=12, s_precision=prec, chain=1, timeout_iters=1)
    with pytest.raises(P.SimrankError) as err:
        h.apply_updates(ups)
        h.sync()
    assert err.value.status == 7
    h.close()
    h = P.SimRank(n, s, d, S0=S0, C=0.6, K=12, s_precision=prec)
    h.apply_updates(ups[:2])
    h.sync()
    want, _ = O.sequential_unit_updates(n, s, d, S0, ups[:2], 0.6, 12)
    assert np.max(np.abs(h.dense() - want)) < (1e-10 if prec == 64 else 1e-6)


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("n,deg,npairs,K", [(300, 6, 1, 5), (300, 6, 2, 1), (300, 6, 1100, 4),
                                            (701, 5, 257, 9), (60, 3, 400, 6)])
def test_gradient_at_block_edges(P, n, deg, npairs, K, weighted):
    """Value and gradient with blocks of two columns and more, repeated pairs and
    pairs of a node with itself, column counts off the padding and off a CTA's 128
    (the quotients before a forward step), nodes without in-links.  Bounds as in
    the adjoint's parity tests."""
    rng = np.random.default_rng(31)
    s, d = degrees_graph(n, [0] + [deg] * (n - 1), 37)
    w = rng.random(s.size).astype(np.float32) + 0.5 if weighted else None
    a, b = rng.integers(0, n, npairs).astype(np.int32), rng.integers(0, n, npairs).astype(np.int32)
    if npairs > 4:
        a[1], b[1], b[2] = a[0], b[0], a[2]
    t = rng.random(npairs)
    sr = P.SimRank(n, s, d, C=0.6, K=K, s_precision=64, mode=1, **({"weight": w} if weighted else {}))
    L, g = sr.grad(a, b, t, s.size)
    L_ref, g_ref, _ = O.pair_loss_and_weight_grad(
        n, s, d, w.astype(np.float64) if weighted else np.ones(s.size), a, b, t, 0.6, K)
    assert abs(L - L_ref) < 1e-11 * max(1.0, abs(L_ref))
    assert np.max(np.abs(g - g_ref)) < 1e-10 * max(1.0, np.max(np.abs(g_ref)))


@pytest.mark.parametrize("K,width", [(15, 908), (15, 909), (15, 1024), (56, 256), (1000, 29)])
def test_fp64_stored_update_over_wide_blocks(P, K, width):
    """FP64 column queries after a stored update: as many columns as one launch of
    its correction holds in shared memory (227 KB, 16 (K + 1) bytes a column),
    one more, a whole block, and long series.  Against Alg 7; 1e-10, as in the
    column-mode parity tests."""
    n, C = 1100, 0.6
    s, d = degrees_graph(n, [0, 1, 40], 41)
    ups = [(next(x for x in range(3, n) if (x, 2) not in set(zip(s.tolist(), d.tolist()))), 2, 1)]
    sr = P.SimRank(n, s, d, C=C, K=K, s_precision=64, mode=P.MODE_COLUMN)
    sr.apply_updates(ups)
    cols = np.random.default_rng(7).choice(n, size=width, replace=False).astype(np.int32)
    got = sr.columns(cols)
    ask = np.unique(np.r_[0, width // 2, width - 2, width - 1])
    base = O.partial_sim_block(O.transition_matrix(n, s, d, sparse=True), cols[ask], K, C)
    for c, q in enumerate(ask.tolist()):
        want = O.inc_sr_all_p(n, s, d, base[:, c], int(cols[q]), ups, C, K)
        assert np.max(np.abs(got[:, q] - want)) < 1e-10


@pytest.mark.parametrize("prec", [64, 32])
def test_s_after_a_wait_that_ran_out(P, prec):
    """One update under bounds of 1 to 2,048 polls: whichever wait of the update
    runs out, in the sums, in the copy of the columns to the panels or in a
    barrier, an entry of S is the old one or the updated one, never a partial
    sum.  1e-10 (FP64) and 1e-6 (FP32), as in the parity tests."""
    n, C, K = 3000, 0.6, 10
    s, d = degrees_graph(n, [0, 1500, 64], 43)
    rng = np.random.default_rng(9)
    S0 = rng.random((n, n))
    S0 = (0.5 * (S0 + S0.T)).astype(np.float64 if prec == 64 else np.float32)
    edges = set(zip(s.tolist(), d.tolist()))
    ups = [(next(x for x in range(3, n) if (x, 1) not in edges), 1, 1)]
    want, _ = O.sequential_unit_updates(n, s, d, S0.astype(np.float64), ups, C, K)
    ran_out = 0
    for limit in [1, 2, 3, 5, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512, 2048]:
        h = P.SimRank(n, s, d, S0=S0, C=C, K=K, s_precision=prec, timeout_iters=limit, s_kernel=1)
        h.apply_updates(ups)
        try:
            h.sync()
        except P.SimrankError as e:
            assert e.status == 7
            ran_out += 1
        got = h.dense()
        h.close()
        err = np.minimum(np.abs(got - S0), np.abs(got - want))
        assert np.max(err) < (1e-10 if prec == 64 else 1e-6), limit
    assert ran_out


@pytest.mark.parametrize("prec,vec", [(64, 0), (32, 0), (32, 1)])
@pytest.mark.parametrize("more", [-1, 0, 1, 700])
def test_recurrence_at_the_switch_between_its_forms(P, prec, vec, more):
    """The flow form takes up to 1,024 nonzeros a CTA; with 5 CTAs the updates
    here go over that number and back, or stay above it.  1e-10 (FP64) and 1e-6
    (FP32), as in the parity tests."""
    n, C, K = 1300, 0.6, 7
    rng = np.random.default_rng(12)
    keys = rng.choice(n * n, 5 * 1024 + more + n, replace=False)
    keys = keys[keys // n != keys % n][: 5 * 1024 + more]
    s, d = (keys // n).astype(np.int32), (keys % n).astype(np.int32)
    edges = set(zip(s.tolist(), d.tolist()))
    ins = [x for x in ((i, j) for i in range(40) for j in (50, 900)) if x not in edges][:3]
    dele = sorted(edges)[100:102]
    ups = [(*ins[0], 1), (*ins[1], 1), (*dele[0], -1), (*dele[1], -1), (*ins[2], 1)]
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-14)
    want, _ = O.sequential_unit_updates(n, s, d, S0, ups, C, K)
    sr = P.SimRank(n, s, d, S0=S0.astype(np.float64 if prec == 64 else np.float32), C=C, K=K,
                   s_precision=prec, vec_fp64=vec, prep_ctas=5)
    sr.apply_updates(ups)
    assert np.max(np.abs(sr.dense() - want)) < (1e-10 if prec == 64 else 1e-6)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("width", [1, 4, 5])
def test_stored_updates_of_rows_that_become_empty(P, prec, width):
    """Stored updates that give an empty in-row and an empty out-row their first
    nonzero and take a row's only one (the chunk lists of narrow steps hold no
    empty rows, those of wide steps end with them), then narrow and wide
    queries.  Against Alg 7: 1e-10 (FP64) and 1e-6 (FP32), as in the column-mode
    parity tests."""
    n, C, K = 140, 0.6, 6
    s, d = degrees_graph(n, [0, 1, 33, 0], 47)
    keep = s != 5  # node 5 has no out-neighbours
    s, d = s[keep], d[keep]
    only = next(x for x in zip(s.tolist(), d.tolist()) if x[1] == 1)
    ups = [(5, 0, 1), (*only, -1), (7, 3, 1), (5, 0, -1), (only[0], 1, 1), (7, 3, -1)]
    cols = np.array([1, 0, 3, 5, 100][:width], np.int32)
    base = O.partial_sim_block(O.transition_matrix(n, s, d, sparse=True), cols, K, C)
    for count in (1, 2, 4, 6):
        sr = P.SimRank(n, s, d, C=C, K=K, s_precision=prec, mode=P.MODE_COLUMN)
        sr.apply_updates(ups[:count])
        got = sr.columns(cols)
        for c, x in enumerate(cols.tolist()):
            want = O.inc_sr_all_p(n, s, d, base[:, c], x, ups[:count], C, K)
            assert np.max(np.abs(got[:, c] - want)) < (1e-10 if prec == 64 else 1e-6), (count, x)


@pytest.mark.parametrize("C", [1e-9, 1e-16, 1e-18, 1e-19, 1e-20, 1e-25, 1e-36, 1e-40, 1e-300])
def test_sweeps_at_a_small_damping_factor(P, C):
    """Sweeps whose factor C / d is near or below the last bit of the fixed-point
    S, for short and long rows: the fixed point and one sweep from another S0.
    Entries are at most 1: 1e-15."""
    n = 300
    s, d = degrees_graph(n, [0, 1, 2, 31, 32, 33, 96, 97, 250, 0], 5)
    Q = O.transition_matrix(n, s, d)
    sr = P.SimRank(n, s, d, C=C, K=1, s_precision=64)
    assert np.max(np.abs(sr.dense() - sweeps(np.eye(n), Q, C, 2))) < 1e-15
    S0 = np.random.default_rng(3).uniform(-1.0, 1.0, (n, n))
    S0 = 0.5 * (S0 + S0.T)
    sr = P.SimRank(n, s, d, S0=S0, C=C, K=1, s_precision=64)
    sr.reanchor(1)
    assert np.max(np.abs(sr.dense() - sweeps(S0, Q, C, 1))) < 1e-15


def test_gradient_of_a_huge_residual(P):
    """Residuals near the largest FP64 number: the quotients before a forward step
    take the division there.  Relative to the largest entry, as in the adjoint's
    parity tests."""
    n, C, K = 60, 0.2, 4
    s, d = degrees_graph(n, [0, 1, 1, 2, 3, 40], 53)
    a, b = np.array([1, 7], np.int32), np.array([5, 1], np.int32)
    t = np.array([-8e307, 0.1])
    sr = P.SimRank(n, s, d, C=C, K=K, s_precision=64, mode=1)
    with np.errstate(over="ignore"):
        L, g = sr.grad(a, b, t, s.size)
        _, want, _ = O.pair_loss_and_weight_grad(n, s, d, np.ones(s.size), a, b, t, C, K)
    assert np.isinf(L) and np.max(np.abs(want)) > 1e305
    assert np.max(np.abs(g / np.max(np.abs(want)) - want / np.max(np.abs(want)))) < 1e-10


@pytest.mark.parametrize("K", [3, 15, 16, 40])
def test_counters_of_the_digit_pass(P, K):
    """tiles_touched and s_bytes count an update's tiles once, however many passes
    of 16 terms its digits take: the numbers of the FP32 CUDA-core pass, with twice
    the bytes."""
    n = 700
    s, d = degrees_graph(n, [0, 5, 64], 59)
    ups = [(x, 0, 1) for x in range(10, 13)]
    nT = (n + 127) // 128
    for aff in (0, 1):
        sr = P.SimRank(n, s, d, C=0.6, K=K, s_precision=64, aff=aff)
        sr.apply_updates(ups)
        st = sr.stats()
        f = P.SimRank(n, s, d, C=0.6, K=K, s_precision=32, s_kernel=1, aff=aff)
        f.apply_updates(ups)
        sf = f.stats()
        assert st["tiles_total"] == sf["tiles_total"] == 3 * nT * (nT + 1) // 2
        assert st["tiles_touched"] == sf["tiles_touched"] <= st["tiles_total"]
        assert st["s_bytes"] == 2 * sf["s_bytes"] and st["panel_bytes"] == 2 * sf["panel_bytes"]


@pytest.mark.parametrize("prec,tc", [(64, 0), (32, 0), (32, 1)])
def test_one_shot_with_an_infinite_block(P, prec, tc):
    """Two graphs without an edge between them, in tiles of their own, S infinite at
    one node of the second: the batch's steps then run in FP64 instead of fixed
    point.  The first graph's block is the oracle's, 1e-10 (FP64) and 1e-6 (FP32)
    as in the one-shot parity tests; the second's is not finite."""
    n, C, K = 128, 0.6, 6
    s, d = degrees_graph(n, [0, 1, 31, 33, 65], 61)
    edges = set(zip(s.tolist(), d.tolist()))
    ups = [(next(x for x in range(9, n) if (x, j) not in edges), j, 1) for j in (0, 4)]
    ups.append((sorted(e for e in edges if e[1] == 3)[0][0], 3, -1))
    new = (edges | {u[:2] for u in ups if u[2] > 0}) - {u[:2] for u in ups if u[2] < 0}
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-15)
    ns, nd = (np.array(v, np.int64) for v in zip(*sorted(new)))
    want = O.one_shot_batch(n, s, d, ns, nd, S0, C, K)
    both = np.zeros((2 * n, 2 * n), np.float64 if prec == 64 else np.float32)
    both[:n, :n] = both[n:, n:] = S0
    both[n + 4, n + 4] = np.inf
    sr = P.SimRank(2 * n, np.r_[s, s + n], np.r_[d, d + n], S0=both, C=C, K=K, s_precision=prec,
                   tc=tc, apply=P.APPLY_ONE_SHOT, relabel=0)
    sr.apply_updates(ups + [(i + n, j + n, op) for i, j, op in ups])
    got = sr.dense()
    assert np.max(np.abs(got[:n, :n] - want)) < (1e-10 if prec == 64 else 1e-6)
    assert not np.all(np.isfinite(got[n:, n:]))


@pytest.mark.parametrize("K", [11, 15])
def test_fp32_digit_pass_rounds_like_fp32(P, K):
    """One update by digits of FP32 panels (FP64 vectors) against the oracle.  A panel
    value is rounded to 2^-24, and C + C^2 + .. < 1.5 of them meet in an entry from
    either vector: 2 * 1.5 * 2 * 2^-24 of the largest |eta|; the four FMAs that join
    the digits and the sum with S round five times more: 11 * 2^-24 of the largest
    entry, of S or of the change."""
    n, C = 5120, 0.6
    s, d = degrees_graph(n, [0, 5, 64], 67)
    S0 = np.random.default_rng(6).random((n, n))
    S0 = (0.5 * (S0 + S0.T)).astype(np.float32)
    edges = set(zip(s.tolist(), d.tolist()))
    ups = [(next(x for x in range(9, n) if (x, 2) not in edges), 2, 1)]
    sr = P.SimRank(n, s, d, S0=S0, C=C, K=K, s_precision=32, vec_fp64=1, aff=0)
    sr.apply_updates(ups)
    want, _ = O.sequential_unit_updates(n, s, d, S0.astype(np.float64), ups, C, K)
    scale = max(np.max(np.abs(want)), np.max(np.abs(want - S0)))
    assert np.max(np.abs(sr.dense() - want)) < 11 * 2.0**-24 * scale


@pytest.mark.parametrize("kw", [{}, {"prep_ctas": 5}])
@pytest.mark.parametrize("scale", [1e-3, 1e-6])
def test_recurrence_of_a_small_s0(P, scale, kw):
    """The part of an update that comes from S0 (the change is affine in S0): from a
    small S0 less the same from S0 = 0.  Entries are of order 1 at most, rounded some
    20 times on either side: 2 * 20 * 2^-53 < 5e-15, far below the part itself."""
    n, C, K = 1300, 0.6, 7
    s, d = degrees_graph(n, [0, 1, 33, 64, 257, 1023], 71)
    edges = set(zip(s.tolist(), d.tolist()))
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-14) * scale
    ups = [(next(x for x in range(9, n) if (x, 1) not in edges), 1, 1)]
    part, ref = [], []
    for start in (S0, np.zeros_like(S0)):
        sr = P.SimRank(n, s, d, S0=start, C=C, K=K, s_precision=64, **kw)
        sr.apply_updates(ups)
        part.append(sr.dense())
        ref.append(O.sequential_unit_updates(n, s, d, start, ups, C, K)[0])
    want = ref[0] - ref[1]
    assert np.max(np.abs(want - S0)) > 1e-2 * scale
    assert np.max(np.abs((part[0] - part[1]) - want)) < 5e-15


@pytest.mark.parametrize("kw", [{}, {"tc": 2, "defer": 4}, {"apply": 1}, {"apply": 2}, {"mode": 1}])
def test_updates_are_not_captured(P, kw):
    """An update on a capturing stream is refused and changes nothing (its sources
    and graph changes lie in memory that the next call rewrites); outside of the
    capture the same update works.  1e-6, as in the parity tests."""
    import torch

    n, C, K = 300, 0.6, 6
    s, d = degrees_graph(n, [0, 1, 33], 73)
    edges = set(zip(s.tolist(), d.tolist()))
    ups = [(next(x for x in range(9, n) if (x, j) not in edges), j, 1) for j in (0, 2)]
    st = torch.cuda.Stream()
    sr = P.SimRank(n, s, d, C=C, K=K, s_precision=32, stream=st.cuda_stream, **kw)
    sr.apply_updates(ups)
    sr.apply_updates([(i, j, -1) for i, j, _ in ups])
    sr.sync()
    before = sr.dense()
    graph = torch.cuda.CUDAGraph()
    buf = torch.zeros(4, device="cuda")
    status = 0
    with torch.cuda.graph(graph, stream=st):
        buf += 1.0
        try:
            sr.apply_updates(ups)
        except P.SimrankError as e:
            status = e.status
    assert status == 6
    assert np.array_equal(sr.dense(), before)
    sr.apply_updates(ups)
    again = P.SimRank(n, s, d, C=C, K=K, s_precision=32, **kw)
    for u in (ups, [(i, j, -1) for i, j, _ in ups], ups):
        again.apply_updates(u)
    assert np.max(np.abs(sr.dense() - again.dense())) < 1e-6


def test_many_graph_updates_are_not_captured(P):
    """The same for many graphs."""
    import torch

    n, C, K = 300, 0.6, 6
    s, d = degrees_graph(n, [0, 1, 33], 73)
    edges = set(zip(s.tolist(), d.tolist()))
    ups = [np.array([(next(x for x in range(9, n) if (x, 2) not in edges), 2, 1)], np.int32)]
    st = torch.cuda.Stream()
    mh = P.MultiSimRank([(n, s, d)], C=C, K=K, s_precision=32, stream=st.cuda_stream)
    before = mh.dense(0)
    graph = torch.cuda.CUDAGraph()
    buf = torch.zeros(4, device="cuda")
    status = 0
    with torch.cuda.graph(graph, stream=st):
        buf += 1.0
        try:
            mh.apply_updates(ups)
        except P.SimrankError as e:
            status = e.status
    assert status == 6
    assert np.array_equal(mh.dense(0), before)
    mh.apply_updates(ups)
    mh.sync()
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-14)
    want, _ = O.sequential_unit_updates(n, s, d, S0, ups[0].tolist(), C, K)
    assert np.max(np.abs(mh.dense(0) - want)) < 1e-6
