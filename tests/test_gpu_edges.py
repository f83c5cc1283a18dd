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
