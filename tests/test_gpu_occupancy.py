"""The vehicles' float32 kernels at 16 and 32 lanes leave room for 512 threads an
SM at every shape that the autotuner offers: their registers stay at 128 or
below, without which full batches run a sixth slower."""
import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [W.pointmass, W.dubins])
def test_threads_an_sm_holds(make):
    import paper_2602_19699_gb300 as P
    P.build()
    prob = make(seed=1)
    b = W.make_batch(prob, 64, seed=2, T=10)
    h = P.tocreate_problem(prob.sys, prob.params, 10)
    rows = [r for r in P.totune(h, b.x0, b.T, P.to_default_opts(prec=P.TO_MIXED, max_iter=1))
            if r["group_lanes"] in (16, 32)]
    assert {r["group_lanes"] for r in rows} == {16, 32}
    for r in rows:
        assert r["ctas_per_sm"] * r["group_lanes"] * r["groups_per_block"] >= 512, r
