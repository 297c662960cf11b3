"""Views of a graph's staging stay valid after the graph object is gone."""
import gc
import weakref

import numpy as np
import pytest

from paper_2602_19699_gb300 import workload as W

pytestmark = pytest.mark.gpu


def test_outputs_outlive_the_graph_object():
    import paper_2602_19699_gb300 as P
    P.build()
    prob = W.pointmass(seed=1)
    h = P.tocreate_problem(prob.sys, prob.params, 20)
    opts = P.to_default_opts(max_iter=2)
    b = W.make_batch(prob, 64, seed=2, T=20)
    g = P.Graph([P.tocreate_batch(h, 64, 64 * 21, opts)], [64], opts=opts)
    x0, T = g.inputs(0)
    x0[:], T[:] = b.x0, b.T
    g.launch()
    g.sync()
    out = g.outputs(0)
    copy = {k: v.copy() for k, v in out.items()}
    owner = weakref.ref(g._staging)
    del g, x0, T
    gc.collect()
    assert owner() is not None               # held by the views
    for k, v in out.items():
        np.testing.assert_array_equal(v, copy[k])
    del out, v
    gc.collect()
    assert owner() is None                   # the last view gives the staging back
