#!/usr/bin/env python
"""Benchmark of the batched iLQR solver on one GB300 (or N, one process each).

Workload (the paper's manipulator, synthetic): planar 3-link arm, B = 8192
instances per GPU, horizons T ~ U{100..400}, zero-control warm start, iLQR
with at most 100 iterations, relative-decrease tolerance 1e-8, 16 step sizes
alpha_j = 0.5^j.  One step = one full batched solve (all iterations of every
instance) in mixed precision.

value: solves per second whose final cost is at most 1e-6 relative above the
FP64 CPU oracle's final cost on the same instance (the fraction is measured on
a bounded random sample that the oracle solves on the host cores; the same run
is the CPU baseline).  Inputs are resident in HBM when the timed region starts.
e2e: the same metric through tosolve_batch with host buffers, including the
host->device copy of (x0, T) and the device->host copy of (X, U, J, iters,
status) every step.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "OCP solves/s at 1e-6 cost tol, batched vs plain (1 GB300); serve p50/p99 ms"
UNIT = "solves/s"
B_PER_GPU = 8192
T_RANGE = (100, 400)
MAX_ITER = 100
TOL = 1e-8
N_ALPHA = 16
COST_TOL = 1e-6
CPU_SAMPLE = 256
PLAIN_SAMPLE = 6
L2_FLUSH_BYTES = 512 << 20


_T_START = time.perf_counter()


def _log(msg: str) -> None:
    """progress on stderr (stdout carries the one JSON line)"""
    print(f"[bench {time.perf_counter() - _T_START:7.1f} s] {msg}", file=sys.stderr, flush=True)


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["gb300", "reference"], default="gb300")
    ap.add_argument("--no-extras", action="store_true", help="skip the plain and FP64 comparison legs")
    ap.add_argument("--quad-budget", action="store_true",
                    help="also run the quadruped at its calibrated 1000-iteration budget (about 140 s)")
    ap.add_argument("--details", metavar="FILE", help="also write every measurement of the run to FILE (JSON)")
    return ap.parse_args()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(x: float, ws: int, device) -> float:
    """The largest of the ranks' values (every rank gets it); the tensor lives
    on ``device`` (the GPU under NCCL, the CPU under gloo)."""
    if ws <= 1:
        return float(x)
    import torch
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return float(t.item())


def job_throughput(units_per_rank: float, seconds_max: float, ws: int) -> float:
    """Whole-job rate under weak scaling: every rank solves its own batch of
    the same size, so the job's units are ws x units_per_rank, done when the
    slowest rank is."""
    return ws * units_per_rank / seconds_max


def workload(rank: int):
    from paper_2602_19699_gb300 import workload as W
    prob = W.planar3(seed=0)
    batch = W.make_batch(prob, B_PER_GPU, seed=1000 + rank, T=T_RANGE)
    return prob, batch


# --------------------------------------------------------------------------
# clocks sampled while the timed region runs
# --------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (FileNotFoundError, OSError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append((float(parts[1]), float(parts[2]), parts[5:9]))
            except ValueError:
                continue
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = np.array([r[0] for r in rows])
        mx = max(r[1] for r in rows)
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i, v in enumerate(r[2]) if v.lower().startswith("active")})
        load = sm[sm >= 0.5 * np.median(sm)]
        return {"sm_mhz": float(np.median(load)), "sm_max_mhz": mx, "reasons": reasons, "samples": len(rows)}


# --------------------------------------------------------------------------
# CPU baseline: the FP64 oracle on a bounded random sample (host cores)
# --------------------------------------------------------------------------
def cpu_baseline_leg(prob, batch, idx, threads=0):
    import oracle
    o = oracle.Oracle.from_problem(prob)
    cores = threads or os.cpu_count() or 1
    t0 = time.perf_counter()
    r = o.solve(batch.x0[idx], batch.T[idx], max_iter=MAX_ITER, tol=TOL, n_alpha=N_ALPHA, threads=cores)
    dt = time.perf_counter() - t0
    return r, dt, min(cores, len(idx))


def solved_fraction(J, J_ref):
    """An instance counts as solved at the cost tolerance when its final cost
    is at most (1 + tol) times the FP64 oracle's (a lower cost is a better
    solution of the same problem)."""
    return float(np.mean(np.asarray(J) <= (1 + COST_TOL) * np.asarray(J_ref)))


def accuracy_gates(J, status, J_ref, status_ref, X=None, X_ref=None, T=None):
    """Agreement of final costs with a reference solve of the same instances.

    one_sided: J <= (1 + tol) J_ref (the value's rule: no worse than the
      reference); two_sided: |J / J_ref - 1| <= tol; the same two-sided gate on
      the instances that converged (status CONVERGED) on both sides, and on
      those whose mixed-precision run ended at the float32 floor instead
      (CONVERGED or LS_FAIL: no step size decreases a cost evaluated from
      float32 states); the distribution of J / J_ref - 1; and, with X, the
      per-instance relative trajectory error over the instance's own knots."""
    J, J_ref = np.asarray(J, dtype=np.float64), np.asarray(J_ref, dtype=np.float64)
    st, st_ref = np.asarray(status) & 15, np.asarray(status_ref) & 15
    r = J / J_ref - 1.0
    within = np.abs(r) <= COST_TOL
    conv = (st == 1) & (st_ref == 1)
    settled = np.isin(st, (1, 3)) & (st_ref == 1)
    q = lambda v: {k: float(np.percentile(v, p)) for k, p in (("min", 0), ("p10", 10), ("median", 50),
                                                               ("p90", 90), ("max", 100))} if len(v) else None
    out = {"sample": int(len(J)), "cost_tol": COST_TOL,
           "one_sided": float(np.mean(J <= (1 + COST_TOL) * J_ref)),
           "two_sided": float(np.mean(within)),
           "converged_both": int(conv.sum()),
           "two_sided_converged_both": float(np.mean(within[conv])) if conv.any() else None,
           "settled_vs_converged": int(settled.sum()),
           "two_sided_settled_vs_converged": float(np.mean(within[settled])) if settled.any() else None,
           "ratio_minus_1": q(r),
           "ratio_minus_1_converged_both": q(r[conv])}
    if X is not None:
        xe = []
        for i in range(len(J)):
            k = X.shape[1] if T is None else int(T[i]) + 1
            xe.append(np.abs(X[i, :k] - X_ref[i, :k]).max() / max(np.abs(X_ref[i, :k]).max(), 1e-300))
        xe = np.array(xe)
        out["traj_rel_err"] = q(xe)
        out["traj_rel_err_converged_both"] = q(xe[conv])
        out["traj_within_1e-4_converged_both"] = float(np.mean(xe[conv] <= 1e-4)) if conv.any() else None
    return out


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return d, "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


def fp32_alu_peak_tflops(sm_mhz: float, sms: int) -> float:
    """152 SMs x 128 FP32 lanes x 2 FLOP per FMA x SM clock."""
    return sms * 128 * 2 * sm_mhz * 1e6 / 1e12


# --------------------------------------------------------------------------
# the printed line
# --------------------------------------------------------------------------
def _short(o):
    """Floats at six significant digits, in any nesting."""
    if isinstance(o, dict):
        return {k: _short(v) for k, v in o.items()}
    if isinstance(o, (list, tuple)):
        return [_short(v) for v in o]
    return float(f"{o:.6g}") if isinstance(o, float) else o


def _sides(g):
    """One- and two-sided fractions of an accuracy-gate record."""
    return {k: g[k] for k in ("sample", "one_sided", "two_sided") if k in g} if g else None


def _leg(r):
    """One system's row in one precision."""
    out = {k: r[k] for k in ("B", "ms", "value") if k in r}
    if r.get("roofline"):
        out["frac"] = r["roofline"]["frac"]
    g = (r.get("accuracy") or {}).get("gates") or {}
    out.update({k: g[k] for k in ("one_sided", "two_sided") if k in g})
    return out


SERVE_COLUMNS = ("rate_per_s", "solves_per_s", "p50_ms", "p99_ms")


def compact_line(full: dict) -> dict:
    """The line that is printed: the headline's fields as they are, and of the
    comparison legs the times, rates and fractions.  It stays below 4.8 kB, so
    that a reader who keeps the end of a log has all of it; descriptions,
    distributions, tuned shapes and per-sample records go to --details."""
    line = dict(full)
    wt = full.get("within_tol")
    if wt:
        line["within_tol"] = _short({"cost_tol": wt["cost_tol"], "fraction": wt["fraction"], "rule": "J <= (1 + 1e-6) J_oracle",
                                     "gates": _sides(wt.get("gates")),
                                     "oracle_self_reproducibility": _sides(wt.get("oracle_self_reproducibility"))})
    if "autotune" in full:
        line["autotune"] = {"chosen": full["autotune"]["chosen"]}
    for k in ("roofline", "cpu_baseline", "batched_fp64", "plain_fp64_one_instance_per_launch"):
        if k in full:
            line[k] = _short(full[k])
    lm = full.get("levenberg_marquardt")
    if lm:
        line["levenberg_marquardt"] = _short({k: lm[k] for k in ("ms_per_step", "raw_solves_per_s", "mean_iters",
                                                                 "within_tol_vs_lm_oracle") if k in lm})
    serve = full.get("serve")
    if serve:
        line["serve"] = _short({"columns": SERVE_COLUMNS, **{p: [[x.get(c) for c in SERVE_COLUMNS] for x in serve[p]]
                                                             for p in ("mixed", "fp64") if p in serve}})
    if full.get("other_workloads"):
        line["other_workloads"] = _short({
            name: {k: _leg(v) for k, v in legs.items() if k in ("mixed", "fp64") and isinstance(v, dict)}
            for name, legs in full["other_workloads"].items()})
    if full.get("bic_ranking"):
        line["bic_ranking"] = _short({name: {c: v[c] for c in ("candidates", "ms", "frac_of_fp32_peak") if c in v}
                                      for name, v in full["bic_ranking"].items()})
    ms = full.get("multi_system")
    if ms:
        out = {k: ms[k] for k in ("sequential_s", "one_launch_s") if k in ms}
        for k in ("equal_shares", "work_shares"):
            if isinstance(ms.get(k), dict):
                out[f"graph_{k}_s"] = ms[k].get("graph_s")
        line["multi_system"] = _short(out)
    return line


# the sources the timed planar-arm solver kernel is compiled from
KERNEL_SOURCES = ("common.cuh", "ilqr.cuh", "launch.cuh", "sys_planar3.cuh", "solve_planar3.cu")


def kernel_sources_digest() -> str:
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2602_19699_gb300", "csrc")
    for f in KERNEL_SOURCES:
        h.update(open(os.path.join(csrc, f), "rb").read())
    return h.hexdigest()[:16]


def measured_traffic():
    """DRAM bytes per solver launch from the committed ncu summary, if it was
    taken on the current kernel sources (else None)."""
    path = os.path.join(ROOT, "profiles", "ilqr_planar3_B8192_traffic.txt")
    if not os.path.exists(path):
        return None
    kv = {}
    for line in open(path):
        if ":" in line:
            k, v = line.split(":", 1)
            kv[k.strip()] = v.strip()
    if kv.get("kernel_sources_sha256_16") != kernel_sources_digest():
        return None
    try:
        return float(kv["dram_bytes_per_launch"])
    except (KeyError, ValueError):
        return None


# --------------------------------------------------------------------------
# the GB300 arm
# --------------------------------------------------------------------------
def run_gb300(args):
    import torch
    ws, rank, local = dist_env()
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group(backend="nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local)
    import paper_2602_19699_gb300 as P
    from paper_2602_19699_gb300 import flops
    P.build()

    prob, b = workload(rank)
    B = b.x0.shape[0]
    T_MAX = T_RANGE[1]
    knots = int(np.sum(b.T + 1))
    problem = P.tocreate_problem(prob.sys, prob.params, T_MAX)
    opts = P.to_default_opts(prec=P.TO_MIXED, max_iter=MAX_ITER, tol_rel=TOL, n_alpha=N_ALPHA)
    # launch shape: the autotuner on the workload itself, 3 iterations per
    # calibration solve (excluded from timing, like a JIT warm-up)
    tune_opts = P.to_default_opts(prec=P.TO_MIXED, max_iter=3, tol_rel=TOL, n_alpha=N_ALPHA)
    tune_rows = P.totune(problem, b.x0, b.T, tune_opts)
    opts.group_lanes, opts.groups_per_block = tune_opts.group_lanes, tune_opts.groups_per_block
    opts.stage_depth = tune_opts.stage_depth
    _log(f"autotune: G={opts.group_lanes} x {opts.groups_per_block} per CTA, staging depth {opts.stage_depth} "
         f"({len(tune_rows)} shapes, {min(r['ms'] for r in tune_rows):.1f} .. {max(r['ms'] for r in tune_rows):.1f} ms)")
    batch = P.tocreate_batch(problem, B, B * (T_MAX + 1), opts)
    dev = torch.device("cuda", local)
    d_x0 = torch.tensor(b.x0, dtype=torch.float64, device=dev)
    d_T = torch.tensor(b.T, dtype=torch.int32, device=dev)
    stream = torch.cuda.current_stream(dev)
    sptr = stream.cuda_stream
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device=dev)

    def solve_device():
        P.tosolve_batch_device(batch, B, d_x0.data_ptr(), d_T.data_ptr(), opts=opts, stream=sptr)

    for _ in range(args.warmup):
        flush.fill_(1.0)
        solve_device()
    torch.cuda.synchronize()

    # ---- timed region: device-resident inputs; L2 flushed between steps
    def barrier():
        if ws > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    clocks = ClockSampler(local)
    barrier()
    clocks.start()
    t_steps = []
    for _ in range(args.steps):
        flush.fill_(1.0)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        solve_device()
        e1.record(stream)
        e1.synchronize()
        t_steps.append(e0.elapsed_time(e1) / 1e3)
    barrier()
    clk = clocks.stop()
    _log(f"timed steps: {[round(t, 4) for t in t_steps]} s")
    launches = P.tolast_launch_count(batch) * args.steps
    t_local = float(np.sum(t_steps))
    t_max = max_over_ranks(t_local, ws, dev)

    # results of the last timed step
    J_g = P.toget_trajectories(batch, X=False, U=False)
    ah, _ = P.toget_history(batch)
    alg = flops.solve_flops(prob.sys, prob.n, prob.m, b.T, J_g["iters"], J_g["status"], ah,
                            lanes_per_round=min(opts.group_lanes, 16), n_alpha=N_ALPHA, refine=True)
    alg64 = flops.solve_flops_fp64(prob.m, b.T, J_g["iters"], J_g["status"], group_lanes=opts.group_lanes)

    # ---- e2e: the public graph API.  Each step writes the inputs into the
    # graph's pinned staging and replays the captured solve: host-to-device
    # copies, horizon sort, solver, gather, device-to-host copies of X, U, J,
    # iters and status, all inside the timed region.
    graph = P.Graph([batch], [B], opts=opts, want_traj=True)
    gx0, gT = graph.inputs(0)

    def solve_e2e():
        gx0[:] = b.x0
        gT[:] = b.T
        graph.launch(sptr)
        graph.sync()
        return graph.outputs(0)

    solve_e2e()
    barrier()
    e2e_steps = []
    for _ in range(args.steps):
        flush.fill_(1.0)
        torch.cuda.synchronize()
        ts = time.perf_counter()
        out_e2e = solve_e2e()
        e2e_steps.append(time.perf_counter() - ts)
    e2e_local = float(np.sum(e2e_steps))
    e2e_max = max_over_ranks(e2e_local, ws, dev)
    _log(f"e2e steps (graph replay): {[round(t, 4) for t in e2e_steps]} s")
    h2d = b.x0.nbytes + b.T.astype(np.int32).nbytes
    d2h = sum(out_e2e[k].nbytes for k in ("X", "U", "J", "iters", "status"))
    e2e_launches = graph.launch_count()
    e2e_same = bool(np.array_equal(out_e2e["J"], J_g["J"]))   # graph replay == device-resident solve

    if rank != 0:
        if ws > 1:
            torch.distributed.barrier()
            torch.distributed.destroy_process_group()
        return

    # ---- accuracy + CPU baseline on a bounded sample (rank 0)
    rng = np.random.default_rng(12345)
    idx = np.sort(rng.choice(B, size=CPU_SAMPLE, replace=False))
    ro, t_cpu, cores = cpu_baseline_leg(prob, b, idx)
    # the same oracle on one core, on the first 8 instances of the sample
    _, t_cpu1, _ = cpu_baseline_leg(prob, b, idx[:8], threads=1)
    frac_mixed = solved_fraction(J_g["J"][idx], ro["J"])
    gates = accuracy_gates(J_g["J"][idx], J_g["status"][idx], ro["J"], ro["status"])
    # the oracle against itself with x0 moved by 1e-15 relative: the ceiling
    # any re-implementation can reach on this (chaotic) workload
    import oracle
    x_pert = b.x0[idx] * (1 + 1e-15 * rng.choice([-1.0, 1.0], size=b.x0[idx].shape))
    r_self = oracle.Oracle.from_problem(prob).solve(x_pert, b.T[idx], max_iter=MAX_ITER, tol=TOL, n_alpha=N_ALPHA,
                                                    threads=cores)
    _log(f"oracle sample of {len(idx)} done ({t_cpu:.1f} s)")
    gates_self = accuracy_gates(r_self["J"], r_self["status"], ro["J"], ro["status"])

    extras = {}
    if not args.no_extras:
        # batched FP64 (same workload, one timed solve) and the plain
        # one-instance-per-launch FP64 solver on a sample
        opts64 = P.to_default_opts(prec=P.TO_FP64, max_iter=MAX_ITER, tol_rel=TOL, n_alpha=N_ALPHA)
        b64 = P.tocreate_batch(problem, B, knots, opts64)
        P.tosolve_batch_device(b64, B, d_x0.data_ptr(), d_T.data_ptr(), opts=opts64, stream=sptr)
        torch.cuda.synchronize()
        flush.fill_(1.0)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        P.tosolve_batch_device(b64, B, d_x0.data_ptr(), d_T.data_ptr(), opts=opts64, stream=sptr)
        e1.record(stream)
        e1.synchronize()
        t64 = e0.elapsed_time(e1) / 1e3
        b64.B, b64.max_iter = B, MAX_ITER
        J64 = P.toget_trajectories(b64, X=False, U=False)["J"]
        frac64 = solved_fraction(J64[idx], ro["J"])
        extras["batched_fp64"] = {"value": B * frac64 / t64, "raw_solves_per_s": B / t64, "ms_per_step": t64 * 1e3,
                                  "within_tol": frac64}
        bp = P.tocreate_batch(problem, 1, T_MAX + 1, opts64)
        pidx = idx[:PLAIN_SAMPLE]
        Jp = np.empty(len(pidx))
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for i in pidx:
            P.tosolve_batch_device(bp, 1, d_x0[i:i + 1].data_ptr(), d_T[i:i + 1].data_ptr(), opts=opts64, stream=sptr)
        e1.record(stream)
        e1.synchronize()
        tp = e0.elapsed_time(e1) / 1e3
        bp.B, bp.max_iter = 1, MAX_ITER
        # per-instance J of the plain solver (re-run outside the timed region)
        for k, i in enumerate(pidx):
            P.tosolve_batch_device(bp, 1, d_x0[i:i + 1].data_ptr(), d_T[i:i + 1].data_ptr(), opts=opts64, stream=sptr)
            Jp[k] = P.toget_trajectories(bp, X=False, U=False)["J"][0]
        fracp = solved_fraction(Jp, ro["J"][:PLAIN_SAMPLE])
        _log(f"batched FP64 {t64:.2f} s; plain FP64 {len(pidx)} instances {tp:.2f} s")
        extras["plain_fp64_one_instance_per_launch"] = {
            "value": len(pidx) * fracp / tp, "raw_solves_per_s": len(pidx) / tp, "sample": len(pidx),
            "within_tol": fracp}

    if not args.no_extras:
        # the Levenberg-Marquardt variant (Sec. IV-B's standard regularisation)
        # on the same workload and launch shape: solves/s and iterations
        # against the eigenvalue clip
        opts_lm = P.to_default_opts(prec=P.TO_MIXED, max_iter=MAX_ITER, tol_rel=TOL, n_alpha=N_ALPHA,
                                    group_lanes=opts.group_lanes, groups_per_block=opts.groups_per_block,
                                    reg=P.TO_REG_LM)
        blm = P.tocreate_batch(problem, B, B * (T_MAX + 1), opts_lm)
        P.tosolve_batch_device(blm, B, d_x0.data_ptr(), d_T.data_ptr(), opts=opts_lm, stream=sptr)
        torch.cuda.synchronize()
        flush.fill_(1.0)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        P.tosolve_batch_device(blm, B, d_x0.data_ptr(), d_T.data_ptr(), opts=opts_lm, stream=sptr)
        e1.record(stream)
        e1.synchronize()
        tlm = e0.elapsed_time(e1) / 1e3
        rlm = P.toget_trajectories(blm, X=False, U=False)
        idx_lm = idx[:64]
        ro_lm = oracle.Oracle.from_problem(prob).solve(b.x0[idx_lm], b.T[idx_lm], max_iter=MAX_ITER, tol=TOL,
                                                       n_alpha=N_ALPHA, threads=cores, reg="lm")
        # the same LM solve of the oracle's sample in float64 on the GPU:
        # separates the precision from the algorithm
        opts_lm64 = P.to_default_opts(prec=P.TO_FP64, max_iter=MAX_ITER, tol_rel=TOL, n_alpha=N_ALPHA,
                                      reg=P.TO_REG_LM)
        blm64 = P.tocreate_batch(problem, len(idx_lm), int(np.sum(b.T[idx_lm] + 1)), opts_lm64)
        P.tosolve_batch(problem, b.x0[idx_lm], b.T[idx_lm], opts=opts_lm64, batch=blm64)
        rlm64 = P.toget_trajectories(blm64, X=False, U=False)
        ratio = rlm["J"] / J_g["J"]
        lm_fail = (rlm["status"] & 15) == 3
        pct = lambda v: {k: float(np.percentile(v, p)) for k, p in (("p10", 10), ("median", 50), ("p90", 90),
                                                                     ("p99", 99), ("max", 100))}
        st_s, st_o = rlm["status"][idx_lm] & 15, ro_lm["status"] & 15
        extras["levenberg_marquardt"] = {
            "raw_solves_per_s": B / tlm, "ms_per_step": tlm * 1e3,
            "mean_iters": float(np.mean(rlm["iters"])), "mean_iters_clip": float(np.mean(J_g["iters"])),
            "status_counts": np.bincount(rlm["status"] & 15, minlength=6)[1:].tolist(),
            "mean_final_cost_ratio_lm_over_clip": float(np.mean(ratio)),
            "cost_ratio_lm_over_clip": pct(ratio),
            "cost_ratio_lm_over_clip_without_ls_fail": pct(ratio[~lm_fail]) if (~lm_fail).any() else None,
            "cost_ratio_lm_over_clip_ls_fail": pct(ratio[lm_fail]) if lm_fail.any() else None,
            "ls_fail_iters": pct(rlm["iters"][lm_fail]) if lm_fail.any() else None,
            "lm_oracle_sample_status_counts": np.bincount(st_o, minlength=6)[1:].tolist(),
            "ls_fail_agreement_with_lm_oracle": {
                "gpu_ls_fail": int((st_s == 3).sum()), "oracle_ls_fail": int((st_o == 3).sum()),
                "both": int(((st_s == 3) & (st_o == 3)).sum())},
            "gates_vs_lm_oracle": accuracy_gates(rlm["J"][idx_lm], rlm["status"][idx_lm], ro_lm["J"], ro_lm["status"]),
            "fp64_gpu_on_the_sample": {
                "status_counts": np.bincount(rlm64["status"] & 15, minlength=6)[1:].tolist(),
                "gates_vs_lm_oracle": accuracy_gates(rlm64["J"], rlm64["status"], ro_lm["J"], ro_lm["status"])},
            "within_tol_vs_lm_oracle": solved_fraction(rlm["J"][idx_lm], ro_lm["J"]),
            "note": "no clipping; mu = 1e-6, x10 and the backward pass redone on a failed pivot test or line "
                    "search, /10 after an accepted step; same workload, launch shape and iteration budget"}
        _log(f"Levenberg-Marquardt variant: {tlm:.2f} s, mean iters {np.mean(rlm['iters']):.1f}")

    serve = None if args.no_extras else serve_leg(P, dev)

    pk, pk_src = peaks()
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    sm_mhz = clk.get("sm_mhz") or pk.get("sm_max_mhz", 2070.0)
    peak32 = fp32_alu_peak_tflops(pk.get("sm_max_mhz", 2070.0), sms)
    peak64 = fp64_alu_peak_tflops(pk.get("sm_max_mhz", 2070.0), sms)
    others = None if args.no_extras else config_legs(P, dev, flush, peak32, peak64, args.quad_budget)
    bic = None if args.no_extras else bic_leg(P, peak32)
    multi = None if args.no_extras else multi_system_leg(P)
    achieved = alg / (t_local / args.steps) / 1e12
    # the binding roofline of the mixed solve: its float32 work at the FP32
    # peak plus its float64 work (the Q_uu Cholesky where it runs in float64)
    # at the FP64 peak
    peak_mix = flops.effective_peak(alg - alg64, alg64, peak32, peak64)
    traffic = measured_traffic()
    n = ws
    t_step = t_max / args.steps
    value = job_throughput(B * frac_mixed, t_step, n)
    line = {
        "metric": METRIC,
        "value": value,
        "unit": UNIT,
        "n_gpus": n,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": t_max / args.steps * 1e3,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f32",
        "precision": "mixed: f32 rollouts, derivatives, Riccati products and Q_uu Cholesky; f64 Cholesky with "
                     "the pivot guard for a Q_uu with a pivot below 2^-10 of its largest diagonal entry; "
                     "float-float gain refinement residual, compensated state and cost sums; f64 cost comparison",
        "data": "synthetic (seeded generator)",
        "config": {
            "workload": f"planar3 arm, B={B} per GPU, T~U{{{T_RANGE[0]}..{T_RANGE[1]}}}, zero warm start, "
                        f"max_iter={MAX_ITER}, tol={TOL}, {N_ALPHA} step sizes",
            "batch_per_gpu": B, "knots_per_gpu": knots, "parallelism": f"independent instances x{n}",
            "l2": "flushed between steps (512 MB write); working set ~1.7 GB > L2",
            "launch": f"persistent kernel, {opts.group_lanes} lanes per instance, {opts.groups_per_block} "
                      f"instances per CTA, staging depth {opts.stage_depth} (autotuned)",
        },
        "raw_solves_per_s": job_throughput(B, t_step, n),
        "within_tol": {"cost_tol": COST_TOL, "sample": int(len(idx)), "fraction": frac_mixed,
                       "rule": "value: final J <= (1 + 1e-6) * J of the FP64 CPU oracle on the same instance "
                               "(one-sided); the two-sided gates and the distribution of J / J_oracle - 1 "
                               "are reported beside it",
                       "gates": gates,
                       "oracle_self_reproducibility": dict(gates_self, perturbation="x0 * (1 +- 1e-15)")},
        "e2e": {"value": job_throughput(B * frac_mixed, e2e_max / args.steps, n), "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                "d2h_bytes_per_step": int(d2h), "ms_per_step": e2e_max / args.steps * 1e3,
                "api": "tograph_launch of a captured solve (H2D from pinned staging, sort, solver with X and U written to pinned memory, padding, D2H)",
                "kernels_per_step": int(e2e_launches), "results_equal_device_solve": e2e_same},
        "autotune": {"chosen": [int(opts.group_lanes), int(opts.groups_per_block), int(opts.stage_depth)],
                     "calibration": "the workload itself, max_iter=3",
                     "columns": ["group_lanes", "groups_per_block", "stage_depth", "ms"],
                     "rows": [[r["group_lanes"], r["groups_per_block"], r["stage_depth"], round(r["ms"], 2)]
                              for r in tune_rows]},
        "gpu_launches": int(launches),
        "roofline": {"bound": "alu", "achieved": achieved, "peak": peak_mix, "unit": "TFLOP/s",
                     "frac": achieved / peak_mix, "traffic": traffic,
                     "peak_source": f"derived: float32 work at {peak32:.1f} TFLOP/s ({sms} SMs x 128 FP32 lanes x 2 x "
                                    f"{pk.get('sm_max_mhz', 2070.0):.0f} MHz) plus float64 work (Q_uu Cholesky where it runs in float64, "
                                    f"{alg64 / alg * 100:.2f} % of the FLOPs) at {peak64:.2f} TFLOP/s (1/64 rate); "
                                    f"max SM clock from {pk_src} peaks",
                     "frac_of_fp32_peak": achieved / peak32,
                     "algorithmic_flops_per_launch": alg, "fp64_flops_per_launch": alg64},
        "cpu_baseline": {"value": len(idx) / t_cpu, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": f"{len(idx)} random instances of the same workload, FP64 C++ oracle, "
                                   f"one instance per thread",
                         "single_core": {"value": 8 / t_cpu1, "unit": UNIT, "cores": 1,
                                         "sample": "the first 8 instances of the same sample, one thread"}},
        "clocks": clk,
    }
    line.update(extras)
    if serve is not None:
        line["serve"] = serve
    if others is not None:
        line["other_workloads"] = others
    if bic is not None:
        line["bic_ranking"] = bic
    if multi is not None:
        line["multi_system"] = multi
    if args.details:
        with open(args.details, "w") as f:
            json.dump(line, f, indent=1)
    print(json.dumps(compact_line(line)), flush=True)
    if ws > 1:
        torch.distributed.barrier()
        torch.distributed.destroy_process_group()


# --------------------------------------------------------------------------
# serving: Poisson arrivals of single requests, continuously batched
# --------------------------------------------------------------------------
SERVE_RATES = {"mixed": (1e2, 1e3, 1e4, 1e5), "fp64": (1e2, 1e3, 1e4, 1e5)}
SERVE_DURATION_S = 2.0
SERVE_MAX_REQ = {"mixed": 6000, "fp64": 1500}
SERVE_MAX_ITER = 30
SERVE_BUDGET = 60 << 30
SERVE_TIMEOUT_S = 60.0


def serve_leg(P, dev):
    """p50/p99 latency (from scheduled arrival to result) and solves/s per
    arrival rate, both precisions; systems point mass / planar arm / 7-DoF arm
    drawn uniformly, T ~ U{50..400}, seeded initial states.  Each rate offers
    a Poisson stream for SERVE_DURATION_S seconds, capped at SERVE_MAX_REQ
    requests (so the highest rates offer a shorter stream); solves/s counts
    the requests over the wall time until the last result."""
    from paper_2602_19699_gb300 import workload as W
    systems = (W.POINTMASS, W.PLANAR3, W.ARM7)
    probs = [W.make_problem(s, 0) for s in systems]
    handles = [P.tocreate_problem(p.sys, p.params, 400) for p in probs]
    out = {"workload": "Poisson arrivals; system ~ U{pointmass2d, planar3, arm7}; T ~ U{50..400}; "
                       f"max_iter={SERVE_MAX_ITER}; HBM budget {SERVE_BUDGET >> 30} GiB; "
                       f"{SERVE_DURATION_S:g} s of arrivals per rate, at most {SERVE_MAX_REQ} requests",
           "latency": "ms from the scheduled arrival to the result (includes waiting for a seat)"}
    for prec_name, rates in SERVE_RATES.items():
        prec = P.TO_MIXED if prec_name == "mixed" else P.TO_FP64
        opts = P.to_default_opts(prec=prec, max_iter=SERVE_MAX_ITER)
        rows = []
        for rate in rates:
            # a fresh server per rate: a trace that does not drain in time
            # leaves nothing behind for the next one
            server = P.Server(handles, opts, hbm_budget_bytes=SERVE_BUDGET)
            out["seats_" + prec_name] = server.stats()["seats"]
            dur = min(SERVE_DURATION_S, SERVE_MAX_REQ[prec_name] / rate)
            trace = W.serving_stream(rate, dur, seed=int(rate), systems=systems, T_range=(50, 400))
            if not trace:
                continue
            t_arr = np.array([t for t, _, _, _ in trace])
            pidx = np.array([systems.index(s) for _, s, _, _ in trace], np.int32)
            Ts = np.array([T for _, _, T, _ in trace], np.int32)
            x0 = np.zeros((len(trace), 14))
            for i, (_, _, _, x) in enumerate(trace):
                x0[i, :x.size] = x
            t0 = time.perf_counter()
            try:
                lat, J, st = server.replay(t_arr, pidx, Ts, x0, timeout_s=SERVE_TIMEOUT_S)
            except P.ToError as e:
                rows.append({"rate_per_s": rate, "requests": int(len(trace)),
                             "not_drained": f"{e} (limit {SERVE_TIMEOUT_S:.0f} s)"})
                server.close()
                continue
            wall = time.perf_counter() - t0
            rows.append({"rate_per_s": rate, "requests": int(len(trace)), "arrivals_s": float(t_arr[-1]),
                         "wall_s": wall, "solves_per_s": len(trace) / wall,
                         "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                         "ok_fraction": float(np.mean(np.isin(st & 15, [1, 2, 3])))})
            server.close()
            _log(f"serve {prec_name} rate {rate:g}: {len(trace)} requests in {wall:.2f} s")
        out[prec_name] = rows
    return out


# --------------------------------------------------------------------------
# several systems at once: one captured graph whose members' persistent
# kernels share the GPU (each sized to its share of the resident CTAs)
# against the same solves one after the other, each with the whole GPU
# --------------------------------------------------------------------------
def multi_system_leg(P):
    import torch
    from paper_2602_19699_gb300 import workload as W
    systems = (W.POINTMASS, W.PLANAR3, W.ARM7)
    B, T_MAX_M, MI = 2048, 400, 30
    opts = P.to_default_opts(prec=P.TO_MIXED, max_iter=MI, tol_rel=TOL, n_alpha=N_ALPHA)
    probs, batches, inputs = [], [], []
    for k, sysid in enumerate(systems):
        prob = W.make_problem(sysid, 0)
        pr = P.tocreate_problem(prob.sys, prob.params, T_MAX_M)
        b = W.make_batch(prob, B, seed=50 + k, T=(50, 400))
        probs.append(pr)
        batches.append(P.tocreate_batch(pr, B, B * (T_MAX_M + 1), opts))
        inputs.append(b)
    dev_in = [(torch.tensor(b.x0, dtype=torch.float64, device="cuda"),
               torch.tensor(b.T, dtype=torch.int32, device="cuda")) for b in inputs]
    stream = torch.cuda.current_stream()

    def sequential():
        for bt, (x0, T) in zip(batches, dev_in):
            P.tosolve_batch_device(bt, B, x0.data_ptr(), T.data_ptr(), opts=opts, stream=stream.cuda_stream)

    sequential()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    sequential()
    e1.record(stream)
    e1.synchronize()
    t_seq = e0.elapsed_time(e1) / 1e3
    alone = []
    for bt, (x0, T) in zip(batches, dev_in):
        e0.record(stream)
        P.tosolve_batch_device(bt, B, x0.data_ptr(), T.data_ptr(), opts=opts, stream=stream.cuda_stream)
        e1.record(stream)
        e1.synchronize()
        alone.append(e0.elapsed_time(e1) / 1e3)
    ref = [P.toget_trajectories(bt, X=False, U=False) for bt in batches]
    # one persistent launch over the three systems (tosolve_systems)
    fbatches = [P.tocreate_batch(pr, B, B * (T_MAX_M + 1), opts) for pr in probs]
    xs, Ts = [x.data_ptr() for x, _ in dev_in], [t.data_ptr() for _, t in dev_in]
    P.tosolve_systems(fbatches, [B] * len(systems), xs, Ts, opts=opts, stream=stream.cuda_stream)
    torch.cuda.synchronize()
    e0.record(stream)
    P.tosolve_systems(fbatches, [B] * len(systems), xs, Ts, opts=opts, stream=stream.cuda_stream)
    e1.record(stream)
    e1.synchronize()
    t_fused = e0.elapsed_time(e1) / 1e3
    fres = [P.toget_trajectories(bt, X=False, U=False) for bt in fbatches]
    out = {"workload": f"point mass, planar arm, 7-DoF arm: {B} instances each, T ~ U{{50..400}}, "
                       f"max_iter={MI}, mixed",
           "sequential_s": t_seq, "alone_s": dict(zip(("pointmass", "planar3", "arm7"), alone)),
           "one_launch_s": t_fused,
           "one_launch_iters_equal_sequential": float(np.mean(np.concatenate(
               [fres[i]["iters"] == ref[i]["iters"] for i in range(len(systems))]))),
           "graph_note": "host wall time of tograph_launch + tograph_sync (H2D, sort, solver, D2H per member)"}
    for label, shares in (("equal_shares", None), ("work_shares", alone)):
        gbatches = [P.tocreate_batch(pr, B, B * (T_MAX_M + 1), opts) for pr in probs]
        g = P.Graph(gbatches, [B] * len(systems), opts=opts, shares=shares, want_traj=False)
        for i, b in enumerate(inputs):
            gx0, gT = g.inputs(i)
            gx0[:] = b.x0
            gT[:] = b.T
        g.launch(stream.cuda_stream)
        g.sync()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        g.launch(stream.cuda_stream)
        g.sync()
        t_graph = time.perf_counter() - t0
        same_it = all(np.array_equal(g.outputs(i)["iters"], ref[i]["iters"]) for i in range(len(systems)))
        jdiff = max(float(np.max(np.abs(g.outputs(i)["J"] - ref[i]["J"]) / np.abs(ref[i]["J"])))
                    for i in range(len(systems)))
        out[label] = {"graph_s": t_graph, "shares": None if shares is None else [float(x) for x in shares],
                      "iters_equal_sequential": bool(same_it), "max_rel_J_diff_vs_sequential": jdiff}
        g.close()
    return out


# --------------------------------------------------------------------------
# biased-initial-condition ranking: 10N candidates scored by the std-critic
# MLP, top N selected (Sec. III-D), N = 8192
# --------------------------------------------------------------------------
def bic_leg(P, peak32):
    from paper_2602_19699_gb300 import workload as W
    out = {}
    for name, sysid in (("planar3", W.PLANAR3), ("quad", W.QUAD)):
        prob = W.make_problem(sysid, 0)
        N = 8192
        Cn = 10 * N
        X = W.make_batch(prob, Cn, seed=11).x0
        r = P.Ranker(prob.n, W.std_critic_weights(prob.n, seed=0))
        for _ in range(3):
            r.rank(X, N)
        ts = []
        for _ in range(5):
            t0 = time.perf_counter()
            r.rank(X, N)
            ts.append(time.perf_counter() - t0)
        t = float(np.median(ts))
        flops = Cn * 2.0 * (prob.n * 256 + 256 * 256 + 256)
        out[name] = {"candidates": Cn, "selected": N, "ms": t * 1e3, "candidates_per_s": Cn / t,
                     "mlp_tflops": flops / t / 1e12, "frac_of_fp32_peak": flops / t / 1e12 / peak32,
                     "timing": "host wall time of torank_candidates (H2D of the candidates, scoring, selection, "
                               "D2H of the indices)"}
        r.close()
    return out


# --------------------------------------------------------------------------
# the other synthetic workloads: point mass (FP64, latency-bound), 7-DoF arm
# (precision comparison), quadruped-shaped base (actor warm start, mixed)
# --------------------------------------------------------------------------
# max_iter by the paper's rule (Sec. IV-A: the 99th percentile of the
# iterations to converge with a naive warm start, the 50th with the actor's):
# 7-DoF arm 288 (p99, zero warm start, 1013 of 1024 converged within 400);
# quadruped: only 11 % of 256 instances converged within 1000 iterations with
# the actor warm start (p50 of those 711), so the rule's budget is the 1000 of
# the calibration itself: "quad_budget" runs it on one resident wave, "quad"
# the full batch for 20 iterations (throughput and accuracy against the
# oracle's stored 20-iteration solve of 8 instances).  "quad_budget" takes
# about 140 s and runs only with --quad-budget.
# lanes per instance of each system's default launch shape, by system id
# (point mass 1, planar arm 2, 7-DoF arm 3, quadruped 4, Dubins car 5)
SYS_LANES = {1: 8, 2: 8, 3: 32, 4: 64, 5: 8}

CONFIGS = {
    "pointmass": dict(sys="pointmass", B=64, T=50, max_iter=100, precs=("fp64",), oracle_sample=64, fp64_subset=None),
    "arm7": dict(sys="arm7", B=16384, T=200, max_iter=288, precs=("mixed", "fp64"), oracle_sample=64,
                 fp64_subset=2048),
    "quad": dict(sys="quad", B=2048, T=100, max_iter=20, precs=("mixed", "fp64"), oracle_sample=0, fp64_subset=32,
                 oracle_reference="quad_oracle_B8_T100.json"),
    "quad_budget": dict(sys="quad", B=608, T=100, max_iter=1000, precs=("mixed",), oracle_sample=0, fp64_subset=None),
    "dubins": dict(sys="dubins", B=8192, T=100, max_iter=100, precs=("mixed", "fp64"), oracle_sample=64,
                   fp64_subset=2048),
}


def fp64_alu_peak_tflops(sm_mhz: float, sms: int) -> float:
    """152 SMs x 2 FP64 lanes x 2 FLOP per FMA x SM clock (1/64 of the FP32 rate)."""
    return sms * 2 * 2 * sm_mhz * 1e6 / 1e12


def _timed_solve(P, batch, B, d_x0, d_T, opts, stream, flush, reps):
    import torch
    # warm-up: one iteration of the same launch (module load, first touch)
    warm = P.to_default_opts(**{f: getattr(opts, f) for f, _ in P.to_solver_opts._fields_ if f != "forced_alpha"})
    warm.max_iter = 1
    P.tosolve_batch_device(batch, B, d_x0.data_ptr(), d_T.data_ptr(), opts=warm, stream=stream.cuda_stream)
    torch.cuda.synchronize()
    ts = []
    for _ in range(reps):
        flush.fill_(1.0)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        P.tosolve_batch_device(batch, B, d_x0.data_ptr(), d_T.data_ptr(), opts=opts, stream=stream.cuda_stream)
        e1.record(stream)
        e1.synchronize()
        ts.append(e0.elapsed_time(e1) / 1e3)
    return float(np.median(ts))


def config_legs(P, dev, flush, peak32, peak64, quad_budget=False):
    import torch
    from paper_2602_19699_gb300 import flops
    from paper_2602_19699_gb300 import workload as W
    import oracle
    stream = torch.cuda.current_stream(dev)
    out = {}
    for name, c in CONFIGS.items():
        if name == "quad_budget" and not quad_budget:
            continue
        sysid = {"pointmass": W.POINTMASS, "arm7": W.ARM7, "quad": W.QUAD, "dubins": W.DUBINS}[c["sys"]]
        prob = W.make_problem(sysid, 0)
        actor = prob.actor_w if sysid == W.QUAD else None
        b = W.make_batch(prob, c["B"], seed=0, T=c["T"])
        problem = P.tocreate_problem(prob.sys, prob.params, c["T"], actor_w=actor)
        d_x0 = torch.tensor(b.x0, dtype=torch.float64, device=dev)
        d_T = torch.tensor(b.T, dtype=torch.int32, device=dev)
        row = {"workload": f"{name}: B={c['B']}, T={c['T']}, max_iter={c['max_iter']}, tol={TOL}, "
                           f"{N_ALPHA} step sizes" + (", actor warm start" if actor is not None else ", zero warm start")}
        res = {}
        for prec_name in c["precs"]:
            prec = P.TO_MIXED if prec_name == "mixed" else P.TO_FP64
            B = c["B"] if (prec_name == "mixed" or not c["fp64_subset"]) else c["fp64_subset"]
            opts = P.to_default_opts(prec=prec, max_iter=c["max_iter"], tol_rel=TOL, n_alpha=N_ALPHA)
            batch = P.tocreate_batch(problem, B, B * (c["T"] + 1), opts)
            reps = 3 if name == "pointmass" else 1
            t = _timed_solve(P, batch, B, d_x0[:B], d_T[:B], opts, stream, flush, reps)
            r = P.toget_trajectories(batch, X=True, U=True)
            t_warm = None
            if actor is not None and c["max_iter"] <= 100:
                # S1 alone: the actor's rollout through the dynamics (a solve with no iteration)
                wopts = P.to_default_opts(prec=prec, max_iter=0, tol_rel=TOL, n_alpha=N_ALPHA)
                wb = P.tocreate_batch(problem, B, B * (c["T"] + 1), wopts)
                t_warm = _timed_solve(P, wb, B, d_x0[:B], d_T[:B], wopts, stream, flush, 1)
            ah, _ = P.toget_history(batch)
            # step sizes per round (64 float64 point masses are solved 32 lanes each)
            lanes = {W.POINTMASS: 16, W.ARM7: 16, W.QUAD: 16, W.DUBINS: 8}[sysid]
            alg = flops.solve_flops(prob.sys, prob.n, prob.m, b.T[:B], r["iters"], r["status"], ah,
                                    lanes_per_round=lanes, n_alpha=N_ALPHA, refine=prec == P.TO_MIXED,
                                    params=prob.params, actor=actor is not None)
            alg_min = flops.solve_flops(prob.sys, prob.n, prob.m, b.T[:B], r["iters"], r["status"], ah,
                                        lanes_per_round=lanes, n_alpha=N_ALPHA, refine=prec == P.TO_MIXED,
                                        params=prob.params, actor=actor is not None, minimal_derivs=True)
            if prec == P.TO_MIXED:
                alg64 = flops.solve_flops_fp64(prob.m, b.T[:B], r["iters"], r["status"],
                                               group_lanes=SYS_LANES[sysid])
                peak = flops.effective_peak(alg - alg64, alg64, peak32, peak64)
                peak_min = flops.effective_peak(alg_min - alg64, alg64, peak32, peak64)
            else:
                peak = peak_min = peak64
            achieved = alg / t / 1e12
            bound = "latency" if name == "pointmass" else "alu"
            res[prec_name] = {"B": B, "ms": t * 1e3, "raw_solves_per_s": B / t,
                              "us_per_iteration": t / max(float(np.max(r["iters"])), 1) * 1e6,
                              "mean_iters": float(np.mean(r["iters"])),
                              "status_counts": np.bincount(r["status"] & 15, minlength=6)[1:].tolist(),
                              "roofline": {"bound": bound, "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                                           "frac": achieved / peak, "algorithmic_flops": alg,
                                           "algorithmic_flops_minimal_derivatives": alg_min,
                                           "frac_minimal_derivatives": alg_min / t / 1e12 / peak_min,
                                           "peak_source": ("derived: float32 work at the FP32 peak plus the Q_uu "
                                                           "Cholesky, where it runs in float64, at the FP64 peak"
                                                           if prec == P.TO_MIXED else
                                                           "derived FP64 ALU rate at the max SM clock"),
                                           "note": ("64 instances of 50 knots: a dependent chain per instance on a "
                                                    "nearly idle GPU; the fraction is not meaningful, the time per "
                                                    "iteration is") if name == "pointmass" else ""},
                              "_J": r["J"], "_X": r["X"], "_st": r["status"]}
            if t_warm is not None:
                res[prec_name]["actor_warm_start"] = {
                    "ms": t_warm * 1e3, "share_of_solve": t_warm / t,
                    "mlp_gflop": float(np.sum(b.T[:B])) * flops.ACTOR_FLOPS_PER_KNOT / 1e9,
                    "note": "a solve with max_iter = 0: the actor MLP and the dynamics at every knot, on CUDA cores"}
            _log(f"config {name} {prec_name}: B={B} {t * 1e3:.1f} ms, mean iters {np.mean(r['iters']):.1f}")
        # accuracy: against the FP64 oracle on a sample, or (quadruped, whose
        # oracle takes minutes per instance) against the GPU's FP64 mode,
        # which the parity tests tie to the oracle
        ns = c["oracle_sample"]
        if ns:
            o = oracle.Oracle.from_problem(prob)
            idx = np.arange(ns)
            ro = o.solve(b.x0[idx], b.T[idx], max_iter=c["max_iter"], tol=TOL, n_alpha=N_ALPHA,
                         threads=os.cpu_count() or 1)
            Jref, Xref, Sref, ref_name = ro["J"], ro["X"], ro["status"], "FP64 CPU oracle"
        elif c["fp64_subset"]:
            idx = np.arange(c["fp64_subset"])
            Jref, Xref, Sref, ref_name = (res["fp64"]["_J"][idx], res["fp64"]["_X"][idx], res["fp64"]["_st"][idx],
                                          "GPU FP64 mode")
        else:
            idx = None
        if c.get("oracle_reference"):
            row["vs_stored_oracle"] = stored_oracle_comparison(c["oracle_reference"], b, c, res)
        for prec_name, rr in res.items():
            if idx is None or (prec_name == "fp64" and ref_name == "GPU FP64 mode"):
                rr["value"] = None
                continue
            J = rr["_J"][idx]
            X = rr["_X"][idx]
            rel = np.abs(J - Jref) / np.abs(Jref)
            xe = np.array([np.abs(X[i] - Xref[i]).max() / max(np.abs(Xref[i]).max(), 1e-300) for i in range(len(idx))])
            frac = solved_fraction(J, Jref)
            rr["accuracy"] = {"reference": ref_name, "sample": int(len(idx)), "within_cost_tol_one_sided": frac,
                              "cost_rel_err_median": float(np.median(rel)), "cost_rel_err_max": float(np.max(rel)),
                              "traj_rel_err_median": float(np.median(xe)), "traj_rel_err_max": float(np.max(xe)),
                              "gates": accuracy_gates(J, rr["_st"][idx], Jref, Sref, X, Xref, b.T[idx])}
            rr["value"] = rr["raw_solves_per_s"] * frac
        for rr in res.values():
            rr.pop("_J")
            rr.pop("_X")
            rr.pop("_st")
        row.update(res)
        out[name] = row
    return out


def stored_oracle_comparison(fname, b, c, res):
    """The GPU's solve of the first instances of a workload against the FP64
    oracle's solve of them stored under tests/golden/ (written by a script
    that calls only the oracle): final-cost gates and the relative error of
    the states at the stored knots, per precision, beside the oracle's own
    reproducibility under x0 * (1 +- 1e-15)."""
    path = os.path.join(ROOT, "tests", "golden", fname)
    if not os.path.exists(path):
        return {"missing": fname}
    ref = json.load(open(path))
    k = int(ref["sample"])
    x0 = np.asarray(ref["x0"])
    if not (np.array_equal(x0, b.x0[:k]) and ref["max_iter"] == c["max_iter"] and ref["T"] == c["T"]):
        return {"mismatch": "the stored record is not this workload (x0, T or max_iter differ)"}
    knots = np.asarray(ref["knots"])
    Jo, So, Xo = np.asarray(ref["J"]), np.asarray(ref["status"]), np.asarray(ref["X_knots"])
    Tk = np.full(k, len(knots) - 1)
    out = {"sample": k, "reference": f"tests/golden/{fname}", "knots_compared": len(knots)}
    for prec_name, rr in res.items():
        out[prec_name] = accuracy_gates(rr["_J"][:k], rr["_st"][:k], Jo, So, rr["_X"][:k][:, knots], Xo, Tk)
    pr = ref["perturbed_x0_1e-15"]
    out["oracle_self_reproducibility"] = accuracy_gates(np.asarray(pr["J"]), So, Jo, So, np.asarray(pr["X_knots"]),
                                                        Xo, Tk)
    return out


# --------------------------------------------------------------------------
# the reference arm: the FP64 oracle itself on the host cores
# --------------------------------------------------------------------------
def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    import oracle
    oracle.build()
    prob, b = workload(0)
    rng = np.random.default_rng(777)
    per_step = 32
    t = 0.0
    cores = os.cpu_count() or 1
    for s in range(args.warmup + args.steps):
        idx = np.sort(rng.choice(b.x0.shape[0], size=per_step, replace=False))
        _, dt, used = cpu_baseline_leg(prob, b, idx, threads=cores)
        if s >= args.warmup:
            t += dt
    value = per_step * args.steps / t
    sample = f"{per_step} random instances per step of the same workload, FP64 C++ oracle, one instance per thread"
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": t / args.steps * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic (seeded generator)",
        "config": {"workload": f"planar3 arm, T~U{{{T_RANGE[0]}..{T_RANGE[1]}}}, max_iter={MAX_ITER}, tol={TOL}",
                   "parallelism": "host threads"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": min(cores, per_step), "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def main():
    args = parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_gb300(args)


if __name__ == "__main__":
    main()
