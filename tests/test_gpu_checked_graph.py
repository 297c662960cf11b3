"""Captured solves on the bounds-checked build (see test_gpu_checked.py): the
solver writes X and U into the graph's staging itself, rows that the checks of
the read-back kernels never see.  Point mass at 8 and 32 lanes, car at 16, planar
arm at 16, the 7-DoF arm (whose rows are gathered) beside them, horizons 1 to
T_max, the staging filled with NaN before.  No violation, and the release
library's results on the same inputs."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def _cases(P, W):
    out, reports = {}, {}
    for name, make, prec, lanes, T_max, B in (("pointmass_8", W.pointmass, P.TO_FP64, 8, 37, 45),
                                              ("pointmass_32", W.pointmass, P.TO_FP64, 32, 37, 45),
                                              ("dubins_16", W.dubins, P.TO_FP64, 16, 37, 45),
                                              ("planar3_16", W.planar3, P.TO_FP64, 16, 37, 45),
                                              ("arm7_32", W.arm7, P.TO_FP64, 32, 9, 5)):
        prob = make(seed=1)
        T = np.resize(np.array([1, T_max, 2, T_max - 1, T_max // 2], np.int32), B)
        h = P.tocreate_problem(prob.sys, prob.params, T_max)
        opts = P.to_default_opts(prec=prec, max_iter=2, group_lanes=lanes)
        g = P.Graph([P.tocreate_batch(h, B, B * (T_max + 1), opts)], [B], opts=opts)
        x0, Ts = g.inputs(0)
        o = g.outputs(0)
        x0[:], Ts[:] = W.make_batch(prob, B, seed=3, T=T_max).x0, T
        o["X"][:], o["U"][:] = np.nan, np.nan
        g.launch()
        g.sync()
        out[name] = {k: np.array(o[k]).tolist() for k in ("X", "U", "J", "status")}
        if P.tobounds_checked():
            reports[name] = P.toget_bounds_report(h, reset=True)
        g.close()
    return out, reports


def _child(path):
    import paper_2602_19699_gb300 as P
    from paper_2602_19699_gb300 import workload as W
    assert P.CHECKED
    P.build()
    assert P.tobounds_checked()
    out, reports = _cases(P, W)
    with open(path, "w") as f:
        json.dump({"results": out, "reports": reports}, f)


@pytest.mark.gpu
def test_captured_solves_stay_in_bounds(tmp_path):
    import paper_2602_19699_gb300 as P
    from paper_2602_19699_gb300 import workload as W
    assert not P.CHECKED
    P.build()
    path = str(tmp_path / "checked.json")
    r = subprocess.run([sys.executable, os.path.abspath(__file__), path], env=dict(os.environ, TO_CHECKED="1"), cwd=ROOT,
                       capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    got = json.load(open(path))
    ref, _ = _cases(P, W)
    assert set(got["reports"]) == set(ref)
    assert not any(v["violations"] for v in got["reports"].values()), got["reports"]
    for name, want in ref.items():
        # the builds may fuse multiply-adds otherwise (test_gpu_checked.py).  The oracle's two iterations move by
        # up to 1.6e-9 of the largest entry when x0 moves by 1e-15; a hundred such roundings a knot stay below 1e-6
        for k in ("X", "U"):
            a, b = np.asarray(got["results"][name][k]), np.asarray(want[k])
            assert np.abs(a - b).max() <= 1e-6 * np.abs(b).max(), (name, k)
        np.testing.assert_allclose(got["results"][name]["J"], want["J"], rtol=1e-9, err_msg=name)
        np.testing.assert_array_equal(np.asarray(got["results"][name]["status"]) & 15, np.asarray(want["status"]) & 15)


if __name__ == "__main__":
    _child(sys.argv[1])
