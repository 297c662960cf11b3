"""Ranking at the edges of its tiles: candidate counts around the tile sizes,
the cluster's ranges and beyond its shared memory.  The selection is exact on
the scores it returns (a stable sort, ties to the lower index), and the scores
agree with the float64 network to 1e-5."""
import numpy as np
import pytest

import oracle
from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2602_19699_gb300 as P
    P.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return P


@pytest.mark.parametrize("n_in", [1, 6, 64])
@pytest.mark.parametrize("C", [1, 15, 16, 17, 127, 129, 255, 2431, 4865, 17025, 19457])
def test_selection_is_exact_on_the_scores(P, n_in, C):
    rng = np.random.default_rng(C)
    w = W.std_critic_weights(n_in, seed=3)
    X = rng.normal(size=(C, n_in))
    X[C // 3:C // 2] = X[0]                               # a run of ties
    r = P.Ranker(n_in, w)
    for N in sorted({1, max(1, C // 10), max(1, C // 2), C}):
        idx, sc = r.rank(X, N, want_scores=True)
        ref = np.sort(np.argsort(-sc, kind="stable")[:N])
        np.testing.assert_array_equal(idx, ref)
    s = oracle.std_critic(w, X[:200])
    np.testing.assert_allclose(sc[:200], s, rtol=1e-5)
    r.close()


def test_more_keys_than_the_cluster_holds(P):
    """700 000 candidates: 87 500 keys a CTA are read from memory each pass; a
    non-finite candidate ranks last."""
    C, N = 700_003, 70_000
    rng = np.random.default_rng(5)
    X = rng.normal(size=(C, 2))
    X[12345] = np.nan
    r = P.Ranker(2, W.std_critic_weights(2, seed=4))
    idx, sc = r.rank(X, N, want_scores=True)
    key = np.where(np.isfinite(sc), sc, 0.0)
    np.testing.assert_array_equal(idx, np.sort(np.argsort(-key, kind="stable")[:N]))
    assert 12345 not in idx
    r.close()
