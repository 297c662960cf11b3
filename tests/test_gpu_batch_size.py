"""A result does not depend on the batch it is solved in: the lanes per
instance that a solve takes for its batch size give the same bits as the
system's default, for both regularisations, a warm start, forced steps and
V_x."""
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


@pytest.mark.parametrize("B", [1, 37])
@pytest.mark.parametrize("reg", ["clip", "lm"])
def test_planar_float32_same_bits_at_8_and_16_lanes(P, B, reg):
    prob = W.planar3(seed=41)
    b = W.make_batch(prob, B, seed=42, T=(1, 60))
    U = np.random.default_rng(1).normal(0, 0.5, (B, 60, prob.m))
    s = P.Solver(prob, T_max=60, prec=P.TO_MIXED, reg=P.TO_REG_LM if reg == "lm" else P.TO_REG_CLIP, max_iter=6)
    want = ("X", "U", "Vx", "K")
    for kw in (dict(), dict(U_init=U), dict(forced_alpha=np.full((B, 6), 3, np.int32))):
        a = s.solve(b.x0, b.T, want=want, want_vx=1, **kw)
        c = s.solve(b.x0, b.T, want=want, want_vx=1, group_lanes=8, **kw)
        for k in ("iters", "status", "alpha_hist", "J", "J_hist", "X", "U", "Vx", "K"):
            np.testing.assert_array_equal(a[k], c[k], err_msg=k)


@pytest.mark.parametrize("make", [W.pointmass, W.dubins])
@pytest.mark.parametrize("B", [1, 37])
@pytest.mark.parametrize("reg", ["clip", "lm"])
def test_vehicles_float64_same_bits_at_8_and_32_lanes(P, make, B, reg):
    prob = make(seed=43)
    b = W.make_batch(prob, B, seed=44, T=(1, 50))
    U = np.random.default_rng(1).normal(0, 0.5, (B, 50, prob.m))
    s = P.Solver(prob, T_max=50, prec=P.TO_FP64, reg=P.TO_REG_LM if reg == "lm" else P.TO_REG_CLIP, max_iter=6)
    want = ("X", "U", "Vx", "K")
    for kw in (dict(), dict(U_init=U), dict(forced_alpha=np.full((B, 6), 3, np.int32))):
        a = s.solve(b.x0, b.T, want=want, want_vx=1, **kw)
        c = s.solve(b.x0, b.T, want=want, want_vx=1, group_lanes=8, **kw)
        for k in ("iters", "status", "alpha_hist", "J", "J_hist", "X", "U", "Vx", "K"):
            np.testing.assert_array_equal(a[k], c[k], err_msg=k)
