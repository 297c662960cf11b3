"""A device allocation that fails is an error of the call that asked for it, and
of no other: what was there before still serves the calls that it is enough
for."""
import ctypes as C

import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2602_19699_gb300 as P
    P.build()
    return P


def test_a_ranker_serves_smaller_requests_after_one_that_does_not_fit(P):
    n_in, C0 = 64, 3000
    X = np.random.default_rng(1).normal(size=(C0, n_in))
    r = P.Ranker(n_in, W.std_critic_weights(n_in, seed=2))
    want = r.rank(X, 100, want_scores=True)
    # 2^31 - 1 candidates of 64 inputs: 1.1 TB, refused before a byte of the input is read
    top, x = np.empty(1, np.int32), np.zeros(1)
    rc = P.lib().torank_candidates(r.handle, 2 ** 31 - 1, x.ctypes.data_as(C.POINTER(C.c_double)), 1,
                                   top.ctypes.data_as(C.POINTER(C.c_int)), None, None)
    assert rc == P.TO_ERR_CUDA
    for n in (C0, 10, C0):
        idx, sc = r.rank(X[:n], min(n, 100), want_scores=True)
        np.testing.assert_array_equal(sc, want[1][:n])
        if n == C0:
            np.testing.assert_array_equal(idx, want[0])
    r.close()


def test_a_batch_solves_after_a_growth_that_does_not_fit(P):
    prob = W.pointmass(seed=1)
    B = 2000
    b = W.make_batch(prob, B, seed=2, T=30)
    h = P.tocreate_problem(prob.sys, prob.params, 30)
    opts = P.to_default_opts(prec=P.TO_FP64, max_iter=3)
    batch = P.tosolve_batch(h, b.x0, b.T, opts=opts)
    want = P.toget_trajectories(batch), P.toget_history(batch)
    opts.max_iter = 2 ** 30                            # histories of 25 TB
    with pytest.raises(P.ToError) as e:
        P.tosolve_batch(h, b.x0, b.T, opts=opts, batch=batch)
    assert e.value.code == P.TO_ERR_CUDA
    opts.max_iter = 3
    got = P.toget_trajectories(P.tosolve_batch(h, b.x0, b.T, opts=opts, batch=batch)), P.toget_history(batch)
    for k in ("X", "U", "J", "iters", "status"):
        np.testing.assert_array_equal(got[0][k], want[0][k], err_msg=k)
    for a, c in zip(got[1], want[1]):
        np.testing.assert_array_equal(a, c)
