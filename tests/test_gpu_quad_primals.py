"""The quadruped's substep primals by teams of lanes against the chains by
single lanes: a mass of 1e-30 kg in a base joint's body sends the same robot to
the latter.  Horizons around the 16 knots that a group's teams take at once and
around its 64 (32) lanes.

Tolerances, relative to the largest entry of an instance's array: the paths
differ in rounding only.  A knot's block is 10 substeps, each a solve with a
mass matrix of condition below 1e5, and the pass multiplies T blocks whose
growth over 40 knots at rest stays below 1e2: 2.2e-16 x 10 x 1e5 x 1e2 = 2e-8
in float64.  In float32 that bound is past 1 beyond a few knots, so the mixed
solves are compared over one and two knots, where no block is multiplied by
more than one other: 6e-8 x 10 x 1e5 x 1e-1 (the errors are not aligned) = 6e-3.
"""
import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [32, 64])
@pytest.mark.parametrize("prec,T,tol", [("fp64", 1, 2e-8), ("fp64", 15, 2e-8), ("fp64", 17, 2e-8), ("fp64", 33, 2e-8),
                                        ("mixed", 1, 6e-3), ("mixed", 2, 6e-3)])
def test_team_primals_equal_the_lane_chains(prec, T, tol, lanes):
    import paper_2602_19699_gb300 as P
    P.build()
    prob = W.quad(seed=1, with_actor=False)
    params = np.array(prob.params, copy=True)
    params[W.RIGID_HEADER + 5] = 1e-30           # the first body's mass
    x0 = W.make_batch(prob, 3, seed=5, T=T).x0
    # one instance's horizon is shorter: its group's teams are partly idle
    Ts = np.array([T, max(1, T - 1), T], np.int32)
    got = []
    for p in (prob.params, params):
        h = P.tocreate_problem(prob.sys, p, T)
        opts = P.to_default_opts(prec=P.TO_FP64 if prec == "fp64" else P.TO_MIXED, max_iter=0, want_vx=1, group_lanes=lanes)
        opts.max_iter = 1
        forced = np.full((3, 1), -1, np.int32)   # no step: the gains and V_x of the warm start
        b = P.tosolve_batch(h, x0, Ts, opts=opts, forced_alpha=forced)
        got.append(P.toget_trajectories(b, Vx=True, K=True))
    for k in ("K", "Vx", "J"):
        a, b = got[0][k], got[1][k]
        for i in range(3):
            assert np.isfinite(a[i]).all() and np.abs(a[i]).max() > 0
            assert np.abs(a[i] - b[i]).max() <= tol * np.abs(b[i]).max(), (k, i, np.abs(a[i] - b[i]).max() / np.abs(b[i]).max())
