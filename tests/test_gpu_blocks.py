"""Derivative blocks kept in the gain records (point mass, Dubins car): V_x and
the gains of one iteration's result against the oracle's backward pass on the
same returned trajectory, at horizons around the group size (a lane with no
knot, one knot, several), every group size and both precisions.

Tolerance: the recursion over T <= 17 knots of n <= 5 states amplifies the unit
roundoff by at most ~ T n kappa(Q_uu) with kappa <= ~30 here (l_uu = 0.01, B^T V
B <= 0.25), 2.6e3 eps: 3e-13 in float64 and 1.5e-4 in float32; the bounds are
1e-11 and 1e-3 of the largest entry."""
import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2602_19699_gb300 as P
    P.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return P


@pytest.mark.parametrize("make", [W.pointmass, W.dubins])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("G", [1, 8, 16, 32])
def test_gains_match_the_oracle(P, oracle_mod, make, prec, G):
    prob = make(seed=31)
    T = np.array([1, 2, 7, 8, 9, 15, 16, 17] * 5, np.int32)
    x0 = W.make_batch(prob, T.size, seed=32, T=1).x0
    s = P.Solver(prob, T_max=17, prec=P.TO_FP64 if prec == "fp64" else P.TO_MIXED, group_lanes=G)
    r = s.solve(x0, T, max_iter=1, tol_rel=0.0, want_vx=1, want=("X", "U", "Vx", "K"))
    o = oracle_mod.Oracle.from_problem(prob)
    tol = 1e-11 if prec == "fp64" else 1e-3
    done = (r["status"] & 15) == P.TO_ST_MAX_ITER       # V_x and K belong to the returned iterate
    assert done[T >= 7].all()       # (the car cannot move its position in one or two knots from rest)
    for i in np.flatnonzero(done):
        t = int(T[i])
        K, _, Vx, rc = o.backward(r["X"][i, :t + 1], r["U"][i, :t])
        assert rc == 0
        assert np.abs(r["K"][i, :t] - K).max() <= tol * np.abs(K).max(), (i, t)
        assert np.abs(r["Vx"][i, :t + 1] - Vx).max() <= tol * np.abs(Vx).max(), (i, t)
