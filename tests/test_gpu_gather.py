"""Read-back of many short instances: a block of the gather holds several, and a
grid that reaches its limit takes more than one set of them.  Every instance's
rows and padding equal the same instance's of a small batch, whose gather has
another shape."""
import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,B,T_max", [(W.pointmass, 2_200_000, 1), (W.pointmass, 70_001, 3), (W.planar3, 20_003, 2),
                                          (W.dubins, 9_001, 17), (W.dubins, 4_099, 40)])
def test_instances_read_back_alike_in_batches_of_any_size(make, B, T_max):
    import paper_2602_19699_gb300 as P
    P.build()
    prob = make(seed=1)
    x0 = W.make_batch(prob, B, seed=3, T=T_max).x0
    T = (1 + np.arange(B) % T_max).astype(np.int32)
    h = P.tocreate_problem(prob.sys, prob.params, T_max)
    opts = P.to_default_opts(prec=P.TO_MIXED, max_iter=1 if B < 1_000_000 else 0, group_lanes=8)
    r = P.toget_trajectories(P.tosolve_batch(h, x0, T, opts=opts))
    some = np.unique(np.concatenate([np.arange(40), B // 2 + np.arange(40), B - 40 + np.arange(40)]))
    q = P.toget_trajectories(P.tosolve_batch(h, x0[some], T[some], opts=opts))
    for k in ("X", "U", "J", "status"):
        np.testing.assert_array_equal(r[k][some], q[k], err_msg=k)
    # every instance: its first row is its state, the rows past its horizon repeat its last and take no control
    np.testing.assert_array_equal(r["X"][:, 0].astype(np.float32), x0.astype(np.float32))
    last = np.take_along_axis(r["X"], T[:, None, None].astype(np.int64), axis=1)
    past = np.arange(T_max + 1)[None, :] >= T[:, None]
    assert np.array_equal(r["X"][past], np.broadcast_to(last, r["X"].shape)[past])
    assert (r["U"][np.arange(T_max)[None, :] >= T[:, None]] == 0).all()
