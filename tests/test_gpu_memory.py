"""Calls whose allocations fail, and what a handle holds afterwards.

An allocation is made to fail on the host: a handle larger than the device's
memory is refused by cudaMalloc at once, and a tensor of PyTorch's takes what is
free but for a few MB."""
import numpy as np
import pytest

from oracle import simrank_oracle as O
from synth import chung_lu_digraph

pytestmark = pytest.mark.gpu

SR_ERR_OOM = 5


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1711_00121_gb300 as P

    return P


def too_large(P):
    """A handle of 1.3 TB of S."""
    e = np.array([0], np.int32), np.array([1], np.int32)
    with pytest.raises(P.SimrankError) as err:
        P.SimRank(400_000, *e, C=0.6, K=1, s_precision=64)
    assert err.value.status == SR_ERR_OOM


class Squeeze:
    """All free device memory but `keep` bytes is taken inside the block."""

    def __init__(self, keep):
        import torch

        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        self.hold = torch.empty(max(1, free - keep), dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        import torch

        self.hold = None
        torch.cuda.empty_cache()


def fixed_point_handle(P, prec, n=2000, **kw):
    C = 0.6
    s, d = chung_lu_digraph(n, 8 * n, 2.1, 2.1, 3)
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-15)
    h = P.SimRank(n, s, d, S0=S0.astype(np.float64 if prec == 64 else np.float32), C=C, K=5,
                  s_precision=prec, **kw)
    return h, S0


@pytest.mark.parametrize("upper", [0, 1])
def test_fp64_s_after_an_error_of_another_call(P, upper):
    """Sweeps of an FP64 S run in its own memory; whatever ends them, S stays the
    matrix it was (here the fixed point, which sweeps keep): 1e-12."""
    h, S0 = fixed_point_handle(P, 64, upper_only=upper)
    too_large(P)
    try:
        h.reanchor(2)
    except P.SimrankError:
        pass
    assert np.max(np.abs(h.dense() - S0)) < 1e-12


@pytest.mark.parametrize("prec", [64, 32])
def test_reanchor_without_memory(P, prec):
    """From too little for the first work buffer to enough for everything: a
    re-anchor works or is refused as out of memory, and S is the fixed point
    either way (1e-12; stored in FP32 1e-6)."""
    h, S0 = fixed_point_handle(P, prec)
    tol = 1e-12 if prec == 64 else 1e-6
    buf = 2048 * 2048 * 8
    refused = 0
    for keep in [buf // 2, 2 * buf - (2 << 20)] + [b * buf + (k << 20) for b in (2, 3)
                                                  for k in (0, 2, 4, 8)]:
        with Squeeze(keep):
            try:
                h.reanchor(2)
            except P.SimrankError as e:
                assert e.status == SR_ERR_OOM, str(e)
                refused += 1
        assert np.max(np.abs(h.dense() - S0)) < tol, keep
    assert refused
    h.reanchor(2)
    assert np.max(np.abs(h.dense() - S0)) < tol


def test_an_error_is_reported_once(P):
    """After a refused handle the calls on other handles work: re-anchor,
    update, query, many graphs."""
    h, S0 = fixed_point_handle(P, 32)
    n = S0.shape[0]
    s, d = chung_lu_digraph(n, 8 * n, 2.1, 2.1, 3)
    mh = P.MultiSimRank([(n, s, d)], C=0.6, K=5, s_precision=32, init_tol=1e-9)
    new = next((x, 7, 1) for x in range(8, n) if (x, 7) not in set(zip(s.tolist(), d.tolist())))
    calls = [lambda: h.reanchor(1), lambda: h.apply_updates([new]), lambda: h.columns([7]),
             lambda: mh.apply_updates([np.array([new], np.int32)]), mh.sync, h.sync]
    for call in calls:
        too_large(P)
        call()
    want, _ = O.sequential_unit_updates(n, s, d, S0, [new], 0.6, 5)
    assert np.max(np.abs(h.columns([7])[:, 0] - want[:, 7])) < 1e-6
    assert np.max(np.abs(mh.columns(0, [7])[:, 0] - want[:, 7])) < 1e-6


@pytest.mark.parametrize("mode", ["dense", "column", "many"])
def test_query_after_a_refused_query(P, mode):
    """A query that is refused for want of memory takes its buffers' capacities
    with it: smaller and equal ones afterwards get memory of their own."""
    n, C, K = 1500, 0.6, 30
    s, d = chung_lu_digraph(n, 8 * n, 2.1, 2.1, 5)
    if mode == "many":
        mh = P.MultiSimRank([(n, s, d)], C=C, K=K, s_precision=32)
        query = lambda cols: mh.columns(0, cols)  # noqa: E731
    else:
        h = P.SimRank(n, s, d, C=C, K=K, s_precision=32, mode=P.MODE_DENSE if mode == "dense" else P.MODE_COLUMN)
        query = h.columns
    want = O.partial_sim_block(O.transition_matrix(n, s, d, sparse=True), np.arange(n), K, C)
    few = np.array([3, 700], np.int32)
    many = np.tile(np.arange(n, dtype=np.int32), 200)  # 3.6 GB of scratch
    for ask in (few, many[:5000], few):
        with Squeeze(64 << 20):
            with pytest.raises(P.SimrankError) as err:
                query(many)
            assert err.value.status == SR_ERR_OOM
        assert np.max(np.abs(query(ask) - want[:, ask])) < 1e-6


@pytest.mark.parametrize("kw", [dict(s_precision=64), dict(s_precision=32, tc=2, defer=2),
                                dict(s_precision=32, tc=2, apply=2), dict(many=1)])
def test_update_without_memory(P, kw):
    """A first update with too little memory for its work buffers is refused, and
    the handle then takes no further updates (the host's graph is ahead of the
    device's) but still answers queries; with enough it gives the oracle's S."""
    n, C, K = 600, 0.6, 1000
    s, d = chung_lu_digraph(n, 8 * n, 2.1, 2.1, 5)
    edges = set(zip(s.tolist(), d.tolist()))
    ups = [(next(x for x in range(n) if x != j and (x, j) not in edges), j, 1) for j in (3, 599)]
    S0 = O.simrank_fixed_point(O.transition_matrix(n, s, d, sparse=True), C, tol=1e-15)
    want, _ = O.sequential_unit_updates(n, s, d, S0, ups, C, K)
    cols = np.array([3, 50, 599], np.int32)
    kw = dict(kw)
    many = kw.pop("many", 0)
    for keep in (6, 10, 14, 20, 30, 40, 400):
        if many:
            h = P.MultiSimRank([(n, s, d)], C=C, K=K, s_precision=32, tc=1)
            apply = lambda: h.apply_updates([np.array(ups, np.int32)])  # noqa: E731
            query = lambda: h.columns(0, cols)  # noqa: E731
        else:
            h = P.SimRank(n, s, d, C=C, K=K, **kw)
            apply, query = lambda: h.apply_updates(ups), lambda: h.columns(cols)  # noqa: E731
        failed = 0
        with Squeeze(keep << 20):
            try:
                apply()
                h.sync()
            except P.SimrankError as e:
                failed = e.status
        h.sync()
        got = query()
        if failed:
            assert failed in (5, 6)
            with pytest.raises(P.SimrankError) as err:
                apply()
            assert "part way" in str(err.value)
        else:
            assert np.max(np.abs(got - want[:, cols])) < (1e-10 if kw.get("s_precision") == 64 else 1e-6)
        h.close()
    assert not failed


def test_kept_buffers_make_room(P):
    """What a re-anchor and queries leave for the next call goes when another
    call, of another handle too, has no room otherwise, and with the last handle."""
    import gc

    import torch

    gc.collect()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    h, S0 = fixed_point_handle(P, 32)
    g, _ = fixed_point_handle(P, 32)
    n = S0.shape[0]
    wide = np.tile(np.arange(n, dtype=np.int32), 3)[:5600]  # 90 MB of scratch
    for _ in range(2):
        h.reanchor(1)  # 3 x 32 MB
        h.columns(np.arange(500, dtype=np.int32))
        with Squeeze(24 << 20):
            assert np.max(np.abs(g.columns(wide) - S0[:, wide])) < 1e-6
        with Squeeze(24 << 20):
            with pytest.raises(P.SimrankError) as err:
                h.reanchor(1)
            assert err.value.status == SR_ERR_OOM
    h.reanchor(1)
    assert np.max(np.abs(h.dense() - S0)) < 1e-6
    h.close()
    g.close()
    torch.cuda.empty_cache()
    # module images and the like stay; three work buffers would be 96 MB
    assert before - torch.cuda.mem_get_info()[0] < 64 << 20


def test_kept_buffers_of_several_threads(P):
    """Handles of four threads, each on a stream of its own, share the kept work
    buffers: re-anchors from the fixed point and queries of several sizes."""
    import threading

    import torch

    made = []
    for t in range(4):
        st = torch.cuda.Stream()
        h, S0 = fixed_point_handle(P, 32, n=900 + 300 * (t // 2), stream=st.cuda_stream)
        made.append((h, S0, st))
    bad = []

    def work(t):
        h, S0, _ = made[t]
        rng = np.random.default_rng(t)
        for _ in range(40):
            if rng.integers(2):
                h.reanchor(int(rng.integers(1, 4)))
            cols = rng.choice(S0.shape[0], int(rng.integers(1, 200)), replace=False).astype(np.int32)
            if not np.max(np.abs(h.columns(cols) - S0[:, cols])) < 1e-6:
                bad.append(t)

    th = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    assert not bad
