"""Critic targets of one batch asked for by several host threads at once, each
with a window of its own: every call has device memory of its own, so each gets
the targets that it gets alone.  With a memory budget that leaves no room beside
the workspace, and with one that does, the same; and a solve that fits the
budget still does after the targets were asked for."""
import threading

import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("budget", ["none", "tight", "roomy"])
def test_threads_get_their_own_targets(budget):
    import paper_2602_19699_gb300 as P
    P.build()
    prob = W.pointmass(seed=5)
    B, T_max, windows = 500, 50, (1, 3, 10, 50)
    b = W.make_batch(prob, B, seed=6, T=(1, T_max))
    h = P.tocreate_problem(prob.sys, prob.params, T_max)
    opts = P.to_default_opts(prec=P.TO_FP64, max_iter=2, want_vx=0)
    knots = B * (T_max + 1)
    if budget != "none":
        # the first budget that the workspace fits in
        lo, hi = 1, 1 << 32
        while lo < hi:
            mid = (lo + hi) // 2
            opts.hbm_budget_bytes = mid
            try:
                P.tosolve_batch(h, b.x0, b.T, opts=opts, batch=P.tocreate_batch(h, B, knots, opts))
                hi = mid
            except P.ToError as e:
                assert e.code == P.TO_ERR_BUDGET
                lo = mid + 1
        opts.hbm_budget_bytes = lo + (0 if budget == "tight" else 16 * B * (T_max + 1))
    batch = P.tosolve_batch(h, b.x0, b.T, opts=opts, batch=P.tocreate_batch(h, B, knots, opts))
    ref = {K: P.toget_critic_targets(batch, K) for K in windows}
    assert not np.array_equal(ref[1], ref[50])
    got, errors = [], []

    def ask(K):
        try:
            for _ in range(50):
                got.append(np.array_equal(P.toget_critic_targets(batch, K), ref[K]))
        except Exception as e:       # pragma: no cover - reported below
            errors.append(e)

    threads = [threading.Thread(target=ask, args=(K,)) for K in windows for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors and len(got) == 50 * len(threads) and all(got)
    # more iterations grow the histories, into what the budget leaves beside the workspace
    if budget != "tight":
        opts.max_iter = 20
        P.tosolve_batch(h, b.x0, b.T, opts=opts, batch=batch)
        opts.max_iter = 2
    P.tosolve_batch(h, b.x0, b.T, opts=opts, batch=batch)
    for K in windows:
        np.testing.assert_array_equal(P.toget_critic_targets(batch, K), ref[K])
