"""Trajectories of a captured solve: written by the solving groups up to each
horizon and padded behind it, or gathered as a whole (single lanes, rigid
trees).  They equal the device-array solve of the same shape bit for bit."""
import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name,lanes", [("pointmass", 1), ("pointmass", 8), ("pointmass", 32), ("dubins", 16),
                                        ("planar3", 8), ("planar3", 16), ("arm7", 32)])
def test_rows_and_padding(name, lanes, prec):
    import paper_2602_19699_gb300 as P
    P.build()
    prob = getattr(W, name)(seed=1)
    T_max, B = 37, 45
    T = np.resize(np.array([1, 37, 2, 36, 17, 37, 5], np.int32), B)
    x0 = W.make_batch(prob, B, seed=3, T=T_max).x0
    h = P.tocreate_problem(prob.sys, prob.params, T_max, actor_w=prob.actor_w)
    opts = P.to_default_opts(prec=P.TO_FP64 if prec == "fp64" else P.TO_MIXED, max_iter=2, group_lanes=lanes)
    g = P.Graph([P.tocreate_batch(h, B, B * (T_max + 1), opts)], [B], opts=opts)
    gx, gT = g.inputs(0)
    out = g.outputs(0)
    ref = P.tosolve_batch(h, x0, T, opts=opts)
    want = P.toget_trajectories(ref)
    for order in (slice(None), slice(None, None, -1)):       # a replay with other horizons leaves nothing behind
        gx[:], gT[:] = x0[order], T[order]
        out["X"][:], out["U"][:] = np.nan, np.nan
        g.launch()
        g.sync()
        for k in ("J", "iters", "status", "X", "U"):
            np.testing.assert_array_equal(out[k], want[k][order], err_msg=k)
    for b in range(B):
        assert (out["U"][B - 1 - b, T[b]:] == 0).all()
        assert (out["X"][B - 1 - b, T[b]:] == out["X"][B - 1 - b, T[b]]).all()
