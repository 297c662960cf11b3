"""A non-finite entry of an initial state ends that instance alone, with the
status of a non-finite cost, whatever the entry: also one that no cost term
sees, like the quadruped's horizontal position.  Every system, entry and
precision, the quadruped at both group sizes and with a base that is a free
body and one that is not; the oracle says the same."""
import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _quad(seed, massive=False):
    prob = W.quad(seed, with_actor=False)
    if massive:
        prob.params = np.array(prob.params, copy=True)
        prob.params[W.RIGID_HEADER + 5] = 1e-30      # the first body's mass: the base is no free body
    return prob


CASES = [("pointmass", W.pointmass, 0), ("dubins", W.dubins, 0), ("planar3", W.planar3, 0), ("arm7", W.arm7, 0)] + [
    (f"{name}_{lanes}", make, lanes) for name, make in (("quad", _quad), ("quad_massive", lambda s: _quad(s, True)))
    for lanes in (32, 64)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name,make,lanes", CASES, ids=[c[0] for c in CASES])
def test_a_non_finite_initial_state_ends_its_instance(oracle_mod, name, make, lanes, prec):
    import paper_2602_19699_gb300 as P
    P.build()
    prob = make(1)
    T = 2
    bad = [(i, v) for i in range(prob.n) for v in (np.nan, np.inf, -np.inf)]
    x0 = W.make_batch(prob, len(bad) + 1, seed=2, T=T).x0
    for k, (i, v) in enumerate(bad):
        x0[k, i] = v
    Ts = np.full(len(x0), T, np.int32)
    h = P.tocreate_problem(prob.sys, prob.params, T)
    opts = P.to_default_opts(prec=P.TO_FP64 if prec == "fp64" else P.TO_MIXED, max_iter=1, tol_rel=0.0, group_lanes=lanes)
    r = P.toget_trajectories(P.tosolve_batch(h, x0, Ts, opts=opts))
    ro = oracle_mod.Oracle.from_problem(prob).solve(x0, Ts, max_iter=1, tol=0.0)
    assert (ro["status"][:-1] == P.TO_ST_NONFINITE).all()
    wrong = [bad[k] for k in range(len(bad)) if r["status"][k] != P.TO_ST_NONFINITE]
    assert not wrong, wrong
    assert r["status"][-1] != P.TO_ST_NONFINITE and np.isfinite(r["J"][-1])   # the others are solved
