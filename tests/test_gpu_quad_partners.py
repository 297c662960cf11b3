"""The quadruped's unforced line search against the oracle on both of its rollout
paths: teams of lanes for a base that is a free body, partner lanes for any
other (a joint offset in the base, inertia or mass in a body that only places
it).  The step sizes are spaced by 0.95, so the accepted ones lie well past the
first lane; the accepted steps, the cost and the trajectory must be the
oracle's.

An instance counts where the oracle's own decisions are clear: every cost that
it compares differs from the current one by more than the margin, 1e-6 of it in
float64 and 1e-3 in float32.  Both are above a cost's rounding: 6 knots of 10
substeps, each a solve of condition below 1e5 whose error enters the state with
the substep's 1e-3 s, 60 x 1e5 x 1e-3 eps = 1.3e-12 and 3.6e-4.  The tolerances
are those of the replays (test_gpu_parity.py): the strict bound, or the
conditioning-scaled one."""
import functools
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W
from test_gpu_parity import FP64_TOL, MIXED_X_TOL, _errors, _inst_rel

pytestmark = pytest.mark.gpu

DECAY, N_ALPHA, T = 0.95, 16, 6


def _robot(kind):
    prob = W.quad(seed=2, with_actor=False)
    p = np.array(prob.params, copy=True)
    body = lambda i: W.RIGID_HEADER + W.BODY_STRIDE * i
    if kind == "offset":
        p[body(4) + 2:body(4) + 5] = (0.03, -0.02, 0.05)
    elif kind == "inertia":
        p[body(3) + 9:body(3) + 12] = (0.02, 0.03, 0.04)
    elif kind == "mass":
        p[body(0) + 5] = 1e-30
    prob.params = p
    return prob


def _margins(o, x0, iters):
    """Smallest relative difference between the current cost and any candidate
    that the oracle's line search looks at."""
    U = np.zeros((T, o.m))
    X, J = o.rollout(x0, U)
    worst = np.inf
    for _ in range(iters):
        K, k, _, _ = o.backward(X, U)
        for j in range(N_ALPHA):
            Xn, Un, Jn = o.forward_pass(X, U, K, k, DECAY ** j)
            worst = min(worst, abs(Jn - J) / J)
            if Jn < J:
                break
        X, U, J = Xn, Un, Jn
    return worst


@functools.lru_cache(maxsize=None)
def _reference(kind, iters):
    """The oracle's solve, its sensitivity to a 1e-15 move of x0 and its margins."""
    import oracle
    prob = _robot(kind)
    b = W.make_batch(prob, 16, seed=1, T=T)
    o = oracle.Oracle.from_problem(prob)
    kw = dict(max_iter=iters, tol=0.0, n_alpha=N_ALPHA, alpha_decay=DECAY)
    ro = o.solve(b.x0, b.T, **kw)
    x1 = b.x0 * (1 + 1e-15 * np.random.default_rng(1).choice([-1.0, 1.0], size=b.x0.shape))
    kappa = _inst_rel(o.solve(x1, b.T, forced=ro["alpha_hist"], **kw)["X"], ro["X"], b.T)
    with ThreadPoolExecutor(16) as ex:
        margins = np.array(list(ex.map(lambda x: _margins(o, x, iters), b.x0)))
    return prob, b, ro, kappa, margins


@pytest.mark.parametrize("kind", ["free", "offset", "inertia", "mass"])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("lanes", [32, 64])
def test_line_search_matches_the_oracle(oracle_mod, kind, lanes, prec):
    import paper_2602_19699_gb300 as P
    P.build()
    iters = 3 if prec == "fp64" else 2
    prob, b, ro, kappa, margins = _reference(kind, iters)
    clear = margins > (1e-6 if prec == "fp64" else 1e-3)
    assert clear.sum() >= 12 and ro["alpha_hist"][clear].max() >= 4     # lanes past the first few decide

    h = P.tocreate_problem(prob.sys, prob.params, T)
    opts = P.to_default_opts(prec=P.TO_FP64 if prec == "fp64" else P.TO_MIXED, max_iter=iters, tol_rel=0.0,
                             n_alpha=N_ALPHA, alpha_decay=DECAY, group_lanes=lanes)
    batch = P.tosolve_batch(h, b.x0, b.T, opts=opts)
    rg = P.toget_trajectories(batch)
    steps, _ = P.toget_history(batch)
    np.testing.assert_array_equal(rg["iters"][clear], iters)
    np.testing.assert_array_equal(steps[clear], ro["alpha_hist"][clear])
    ex, ej = _errors(ro, rg, b.T)
    tol, scale = (FP64_TOL, 1e3) if prec == "fp64" else (MIXED_X_TOL, 1e11)
    bound = np.maximum(tol, scale * kappa)
    assert np.all(ex[clear] <= bound[clear]), (ex[clear], kappa[clear])
    assert np.all(ej[clear] <= bound[clear]), (ej[clear], kappa[clear])
