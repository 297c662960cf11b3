"""The work a user of this package has it do, as cases that can be timed.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (problem handles, workspaces, inputs from the seed), ``run``
is one pass through the public entry points, ``work`` counts what the pass
cannot do without and ``exact`` computes its outputs in 64 bits in plain
torch, without this package's solver.

Kinds of case:

* ``solve``: a batch of trajectory optimisations with a fixed iteration
  budget.  ``entry`` says how the program calls: ``noalloc`` (device tensors
  in and out, nothing allocated: a control loop), ``solver`` (host arrays
  through ``Solver.solve``: data collection, with the accepted steps, V_x, the
  gains K and the critic targets of a ``window`` where asked for) or ``graph``
  (a captured solve with pinned staging: a long-running loop over batches).
* ``rank``: the choice of the N most promising of C candidate starts.

``prec`` is the arithmetic of the solve.  Results of a float32 ("mixed")
solve go on as float32 tensors on the GPU, the type in which the networks
that consume them train; float64 results stay float64.

Horizons and budgets are those at which two correct solvers can be compared:
the arms are chaotic (float64 rounding grows by 1e4 and more within 50 knots,
float32 rounding past any use within 20), so their float64 cases are short
control horizons, and their float32 ones, at planning length, have no value in
64 bits (``exact`` gives None).
"""
import math

import numpy as np
import torch

import paper_2602_19699_gb300 as P
from paper_2602_19699_gb300 import flops as F
from paper_2602_19699_gb300 import workload as W

SYS = {"pointmass": W.POINTMASS, "planar3": W.PLANAR3, "arm7": W.ARM7, "quad": W.QUAD, "dubins": W.DUBINS}
N_ALPHA, DECAY, EPS = 16, 0.5, 1e-8      # the solver's defaults


def _solve(system, prec, B, T, iters, entry, vx=False, window=0):
    return {"kind": "solve", "system": system, "prec": prec, "B": B, "T_lo": T[0], "T_hi": T[1], "iters": iters,
            "entry": entry, "vx": vx, "window": window}


def listed():
    return [
        # one vehicle replanned in a control loop: the smallest call
        dict(_solve("pointmass", "fp64", 1, (50, 50), 2, "noalloc"), name="pointmass_control"),
        # the point-mass configuration of the bench, 64 starts
        dict(_solve("pointmass", "fp64", 64, (50, 50), 2, "solver"), name="pointmass_batch"),
        # training data for the car: solutions, V_x, gains and critic targets
        dict(_solve("dubins", "fp64", 2048, (100, 100), 3, "solver", True, 20), name="dubins_collect"),
        # the car's large batch, replayed with new starts and horizons
        dict(_solve("dubins", "mixed", 8192, (20, 50), 2, "graph"), name="dubins_large"),
        # one arm replanned in a control loop
        dict(_solve("planar3", "mixed", 1, (100, 100), 3, "noalloc"), name="planar3_control"),
        # a medium batch of the arm, ragged horizons
        dict(_solve("planar3", "mixed", 613, (100, 400), 3, "solver"), name="planar3_medium"),
        # the bench's workload: 8192 arms, horizons 100 to 400
        dict(_solve("planar3", "mixed", 8192, (100, 400), 5, "graph"), name="planar3_bench"),
        # the arm in float64 over short control horizons, with V_x, gains and critic targets
        dict(_solve("planar3", "fp64", 1024, (10, 20), 2, "solver", True, 8), name="planar3_fp64"),
        # the 7-DoF arm's large batch
        dict(_solve("arm7", "mixed", 2048, (50, 200), 2, "graph"), name="arm7_large"),
        # the 7-DoF arm in float64 over short control horizons
        dict(_solve("arm7", "fp64", 304, (10, 20), 2, "solver", True, 8), name="arm7_fp64"),
        # the quadruped with the actor's warm start: one iteration a tick over a short horizon
        dict(_solve("quad", "mixed", 512, (4, 8), 1, "solver", True), name="quad_mpc"),
        # the biased choice of initial conditions: 8192 starts out of 81 920
        {"kind": "rank", "system": "planar3", "C": 81920, "N": 8192, "name": "rank_81920"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    kind = rng.choice(["pointmass", "dubins", "dubins32", "planar32", "planar32", "planar64", "arm32", "arm64", "quad32", "quad64",
                       "rank", "rank"])
    if kind == "rank":
        C = _log(rng, 700, 81920)
        return {"kind": "rank", "system": rng.choice(["pointmass", "planar3", "arm7", "quad"]), "C": C, "N": max(1, C // 10)}
    if kind == "pointmass":
        B = _log(rng, 1, 1024)
        return _solve("pointmass", "fp64", B, (rng.randint(10, 49), 50), rng.randint(1, 2), rng.choice(["solver", "noalloc"]))
    if kind == "dubins":
        T = rng.randint(20, 100)
        return _solve("dubins", "fp64", _log(rng, 8, 2048), (max(10, T // 2), T), rng.randint(1, 3), "solver", True, rng.randint(1, T))
    if kind == "dubins32":
        return _solve("dubins", "mixed", _log(rng, 100, 16384), (20, rng.randint(21, 50)), rng.randint(1, 2), rng.choice(["graph", "solver"]))
    if kind == "planar32":
        B, T = _log(rng, 1, 8192), rng.randint(50, 400)
        entry = rng.choice(["noalloc", "solver"]) if B <= 64 else rng.choice(["graph", "solver"])
        return _solve("planar3", "mixed", B, (T // 2, T), rng.randint(1, 5), entry)
    if kind == "planar64":
        T = rng.randint(6, 20)
        return _solve("planar3", "fp64", _log(rng, 1, 3000), (max(1, T // 2), T), rng.randint(1, 2), "solver", True, rng.randint(1, 10))
    if kind == "arm32":
        T = rng.randint(20, 200)
        return _solve("arm7", "mixed", _log(rng, 1, 2048), (T // 2, T), rng.randint(1, 2), rng.choice(["graph", "solver"]))
    if kind == "arm64":
        T = rng.randint(6, 20)
        return _solve("arm7", "fp64", _log(rng, 1, 608), (max(1, T // 2), T), rng.randint(1, 2), "solver", True, rng.randint(1, 10))
    if kind == "quad32":
        T = rng.randint(3, 8)
        return _solve("quad", "mixed", _log(rng, 1, 1000), (max(1, T // 2), T), 1, rng.choice(["graph", "solver"]))
    return _solve("quad", "fp64", _log(rng, 1, 64), (3, rng.randint(5, 8)), 1, "solver", True)


def _inputs(case, seed):
    """The problem (fixed, as a program's is) and the seed's initial states and horizons."""
    prob = W.make_problem(SYS[case["system"]], seed=0)
    b = W.make_batch(prob, case["B"], seed=seed, T=(case["T_lo"], case["T_hi"]))
    return prob, b.x0, b.T


def _candidates(case, seed):
    prob = W.make_problem(SYS[case["system"]], seed=0)
    return W.make_batch(prob, case["C"], seed=seed, T=1).x0, W.std_critic_weights(prob.n, seed=0)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "rank":
        s["x"], w = _candidates(case, seed)
        s["ranker"] = P.Ranker(s["x"].shape[1], w)
        return s
    prob, x0, T = _inputs(case, seed)
    prec = P.TO_FP64 if case["prec"] == "fp64" else P.TO_MIXED
    opts = dict(max_iter=case["iters"], tol_rel=0.0, want_vx=int(case["vx"]))
    B, T_max = case["B"], case["T_hi"]
    if case["entry"] == "solver":
        s["solver"] = P.Solver(prob, T_max=T_max, prec=prec, B_max=B, **opts)
        s["x0"], s["T"] = x0, T
        return s
    s["problem"] = P.tocreate_problem(prob.sys, prob.params, T_max, actor_w=prob.actor_w)
    s["opts"] = P.to_default_opts(prec=prec, **opts)
    if case["entry"] == "graph":
        s["graph"] = P.Graph([P.tocreate_batch(s["problem"], B, B * (T_max + 1), s["opts"])], [B], opts=s["opts"])
        gx, gT = s["graph"].inputs(0)
        gx[:], gT[:] = x0, T
        return s
    f8, i4 = dict(dtype=torch.float64, device="cuda"), dict(dtype=torch.int32, device="cuda")
    s["x0"], s["T"] = torch.from_numpy(x0).cuda(), torch.from_numpy(T).cuda()
    s["out"] = {"J": torch.empty(B, **f8), "iters": torch.empty(B, **i4), "status": torch.empty(B, **i4),
                "X": torch.empty((B, T_max + 1, prob.n), **f8), "U": torch.empty((B, T_max, prob.m), **f8)}
    return s


def _given(out, prec):
    """The results that were asked for; a float32 solve's as the float32 GPU tensors that training takes."""
    out = {k: v for k, v in out.items() if v is not None}
    if prec == "mixed":
        out = {k: (torch.as_tensor(v).cuda().float() if str(v.dtype).endswith("float64") else v) for k, v in out.items()}
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "rank":
        idx, scores = state["ranker"].rank(state["x"], case["N"], want_scores=True)
        return {"idx": idx, "scores": scores}
    if case["entry"] == "solver":
        out = state["solver"].solve(state["x0"], state["T"], want=("X", "U", "Vx", "K") if case["vx"] else ("X", "U"))
        if case["window"]:
            out["Vbar"] = P.toget_critic_targets(state["solver"].batch, case["window"])
    elif case["entry"] == "graph":
        state["graph"].launch()
        state["graph"].sync()
        out = state["graph"].outputs(0)
    else:
        out = state["out"]
        P.tosolve_batch_noalloc(state["problem"], case["B"], state["x0"].data_ptr(), state["T"].data_ptr(),
                                out["J"].data_ptr(), out["iters"].data_ptr(), out["status"].data_ptr(), out["X"].data_ptr(),
                                out["U"].data_ptr(), opts=state["opts"], stream=torch.cuda.current_stream().cuda_stream)
    return _given(out, case["prec"])


def work(case):
    """Each input read and each output written once; per knot one rollout of the warm start and, per iteration, one
    linearisation by analytic derivatives, one Riccati step and one accepted candidate."""
    if case["kind"] == "rank":
        n = W.NM[SYS[case["system"]]][0]
        C, H = case["C"], 256
        return {"bytes": C * (8 * n + 4) + 4 * case["N"] + 4 * (H * n + H * H + 3 * H + 1), "flops": 2.0 * C * (H * n + H * H + H)}
    prob = W.make_problem(SYS[case["system"]], seed=0)
    n, m, B, T_max = prob.n, prob.m, case["B"], case["T_hi"]
    knots = B * (case["T_lo"] + T_max) / 2
    roll = F.rollout_flops(prob.sys, n, m, prob.params)
    lin = F.derivative_flops_minimal(prob.sys, n, m, prob.params) + F.riccati_flops(n, m, case["prec"] == "mixed")
    flops = roll + case["iters"] * (lin + roll) + (lin if case["vx"] else 0)
    if prob.actor_w is not None:
        flops += F.ACTOR_FLOPS_PER_KNOT
    out = (T_max + 1) * n + T_max * m + 1
    if case["vx"]:
        out += (T_max + 1) * n + T_max * m * n
    if case["window"]:
        out += T_max + 1
    return {"bytes": B * (8 * (n + out) + 12), "flops": flops * knots}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _bumps(x, p):
    nb = int(p[4])
    c = torch.as_tensor(np.asarray(p[5:5 + 2 * nb]).reshape(nb, 2), dtype=x.dtype, device=x.device)
    d = x[..., None, :2] - c
    return (p[2] * torch.exp(-(d * d).sum(-1) / (2 * p[3] ** 2))).sum(-1)


class _PointMass:
    def __init__(self, p):
        self.p, self.k = p, 5 + 2 * int(p[4])

    def f(self, x, u):
        return torch.cat([x[..., :2] + self.p[0] * x[..., 2:], x[..., 2:] + self.p[0] * u], -1)

    def l(self, x, u):
        return self.p[1] * (u * u).sum(-1) + _bumps(x, self.p)

    def lT(self, x):
        return self.p[self.k] * (x[..., :2] ** 2).sum(-1) + self.p[self.k + 1] * (x[..., 2:] ** 2).sum(-1)


class _Dubins(_PointMass):
    def f(self, x, u):
        dt, v = self.p[0], x[..., 3]
        return torch.stack([x[..., 0] + dt * v * torch.cos(x[..., 2]), x[..., 1] + dt * v * torch.sin(x[..., 2]),
                            x[..., 2] + dt * u[..., 0], v + dt * x[..., 4], x[..., 4] + dt * u[..., 1]], -1)

    def lT(self, x):
        return self.p[self.k] * (x[..., :2] ** 2).sum(-1) + self.p[self.k + 1] * x[..., 3] ** 2 + self.p[self.k + 2] * x[..., 4] ** 2


class _Tree:
    """A tree of one-axis joints; inverse dynamics by Newton and Euler's equations in each body's own frame."""

    def __init__(self, prob):
        p = prob.params
        self.p, self.N, self.kind = p, int(p[4]), prob.sys
        self.bodies = np.asarray(p[8:8 + 16 * self.N]).reshape(self.N, 16)
        self.c = p[8 + 16 * self.N:]
        self.a0, self.n_sub = int(p[5]), max(1, int(p[6]))

    @staticmethod
    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

    def rot(self, i, q, v, back):
        """v from the parent's axes to body i's (back: the other way)"""
        a = int(self.bodies[i, 1])
        if a > 2:
            return list(v)
        j, k = (a + 1) % 3, (a + 2) % 3
        c, s = torch.cos(q), torch.sin(q)
        s = -s if back else s
        r = [None] * 3
        r[a], r[j], r[k] = v[a] + 0 * c, c * v[j] + s * v[k], c * v[k] - s * v[j]
        return r

    def place(self, i, q):
        """body i's origin in its parent's axes"""
        r = [q * 0 + t for t in self.bodies[i, 2:5]]
        a = int(self.bodies[i, 1])
        if a > 2:
            r[a - 3] = r[a - 3] + q
        return r

    def chain(self, i):
        out = []
        while i >= 0:
            out.append(i)
            i = int(self.bodies[i, 0])
        return out

    def world(self, i, q, v, point):
        """body i's vector (a point of it) in world axes"""
        for j in self.chain(i):
            v = self.rot(j, q[..., j], v, True)
            if point:
                v = [x + y for x, y in zip(v, self.place(j, q[..., j]))]
        return v

    def inverse(self, q, qd, qdd, on, contact):
        """the joint forces; gravity and contact count where on is 1"""
        cr, z = self.cross, 0 * q[..., 0]
        add = lambda *v: [sum(t) for t in zip(*v)]  # noqa: E731
        w, wd, a, v, f, n, rs = ([None] * self.N for _ in range(7))
        for i in range(self.N):
            b, pa, jt = self.bodies[i], int(self.bodies[i, 0]), int(self.bodies[i, 1])
            r = rs[i] = self.place(i, q[..., i])
            pw, pwd, pv = (w[pa], wd[pa], v[pa]) if pa >= 0 else ([z] * 3, [z] * 3, [z] * 3)
            p_a = a[pa] if pa >= 0 else [z - g * on for g in self.p[1:4]]
            turn = lambda t: self.rot(i, q[..., i], t, False)  # noqa: E731, B023
            w[i], wd[i] = turn(pw), turn(pwd)
            v[i], a[i] = turn(add(pv, cr(pw, r))), turn(add(p_a, cr(pwd, r), cr(pw, cr(pw, r))))
            s = [z] * 3
            if jt < 3:
                s[jt] = qd[..., i]
                wd[i] = add(wd[i], cr(w[i], s))
                w[i][jt], wd[i][jt] = w[i][jt] + qd[..., i], wd[i][jt] + qdd[..., i]
            else:
                s[jt - 3] = qd[..., i]
                a[i] = [x + 2 * y for x, y in zip(a[i], cr(w[i], s))]
                v[i][jt - 3], a[i][jt - 3] = v[i][jt - 3] + qd[..., i], a[i][jt - 3] + qdd[..., i]
            com = b[6:9]
            f[i] = [b[5] * t for t in add(a[i], cr(wd[i], com), cr(w[i], cr(w[i], com)))]
            n[i] = add([I * t for I, t in zip(b[9:12], wd[i])], cr(w[i], [I * t for I, t in zip(b[9:12], w[i])]), cr(com, f[i]))
        if contact:
            kc, dc, beta = self.c[7:10]
            for t in range(int(self.c[10])):
                i, pt = int(self.c[11 + 4 * t]), list(self.c[12 + 4 * t:15 + 4 * t])
                height = self.world(i, q, [z + t for t in pt], True)[2]
                vel = self.world(i, q, add(v[i], cr(w[i], pt)), False)
                gate = torch.sigmoid(-beta * height)
                F_ = [-dc * on * gate * x for x in vel]
                F_[2] = F_[2] + kc * on * torch.nn.functional.softplus(-height, beta=float(beta), threshold=600.0)
                for j in reversed(self.chain(i)):
                    F_ = self.rot(j, q[..., j], F_, False)
                f[i] = [x - y for x, y in zip(f[i], F_)]
                n[i] = [x - y for x, y in zip(n[i], cr(pt, F_))]
        tau = [None] * self.N
        for i in range(self.N - 1, -1, -1):
            pa, jt = int(self.bodies[i, 0]), int(self.bodies[i, 1])
            tau[i] = n[i][jt] if jt < 3 else f[i][jt - 3]
            if pa >= 0:
                g, m = self.rot(i, q[..., i], f[i], True), self.rot(i, q[..., i], n[i], True)
                f[pa], n[pa] = add(f[pa], g), add(n[pa], m, cr(rs[i], g))
        return torch.stack(tau, -1)

    def f(self, x, u):
        N, h = self.N, self.p[0] / self.n_sub
        q, qd = x[..., :N], x[..., N:]
        tau = torch.cat([0 * q[..., :self.a0], u], -1)
        # N unit accelerations at rest give the mass matrix, row N at no acceleration the bias
        unit = torch.eye(N + 1, dtype=x.dtype, device=x.device)
        for _ in range(self.n_sub):
            qe, qde = (t[..., None, :].expand(*t.shape[:-1], N + 1, N) for t in (q, qd))
            r = self.inverse(qe, qde * unit[:, N:], unit[:, :N] + 0 * qe, unit[:, N], self.kind == W.QUAD)
            qd = qd + h * torch.linalg.solve(r[..., :N, :], (tau - r[..., N, :])[..., None])[..., 0]
            q = q + h * qd
        return torch.cat([q, qd], -1)

    def ee(self, x):
        pt = self.c[13:16] if self.kind == W.PLANAR3 else self.c[8:11]
        return torch.stack(self.world(self.N - 1, x, [0 * x[..., 0] + t for t in pt], True), -1)

    def base(self, x):
        c = self.c
        return c[2] * (x[..., 2] - c[1]) ** 2 + c[3] * (x[..., 3:6] ** 2).sum(-1) + c[4] * (x[..., 18] - c[5]) ** 2

    def l(self, x, u):
        c = self.c
        s = c[0] * (u * u).sum(-1)
        if self.kind == W.QUAD:
            return s + self.base(x)
        if self.kind == W.ARM7:
            return s + c[1] * (x[..., self.N:] ** 2).sum(-1)
        nb = int(c[3])
        d = self.ee(x)[..., None, :2] - torch.as_tensor(np.array(c[4:4 + 2 * nb]).reshape(nb, 2), device=x.device)
        return s + (c[1] * torch.exp(-(d * d).sum(-1) / (2 * c[2] ** 2))).sum(-1)

    def lT(self, x):
        c = self.c
        if self.kind == W.QUAD:
            return c[6] * self.base(x)
        t, wee, wv = (c[8:10], c[10], c[11]) if self.kind == W.PLANAR3 else (c[2:5], c[5], c[6])
        d = self.ee(x)[..., :len(t)] - torch.as_tensor(np.array(t), device=x.device)
        return wee * (d * d).sum(-1) + wv * (x[..., self.N:] ** 2).sum(-1)


def _actor(w, x):
    n, m = 36, 12
    W1, b1, W2, b2, W3, b3 = torch.split(torch.from_numpy(w).double().to(x.device), [256 * n, 256, 256 * 256, 256, 256 * m, m])
    h = torch.tanh(x @ W1.reshape(256, n).T + b1)
    return torch.tanh(h @ W2.reshape(256, 256).T + b2) @ W3.reshape(m, 256).T + b3


def _clip(H):
    """max(eigenvalue, eps), the eigenvectors kept"""
    s, V = torch.linalg.eigh(H.cpu())
    return ((V * s.clamp_min(EPS)[..., None, :]) @ V.mT).to(H.device)


def _chunks(fn, *a, size=1 << 15):
    parts = [torch.func.vmap(fn)(*(t[i:i + size] for t in a)) for i in range(0, a[0].shape[0], size)]
    return torch.cat(parts) if torch.is_tensor(parts[0]) else tuple(torch.cat(c) for c in zip(*parts))


def _ilqr(sysm, x0, T, m, iters, vx, window, actor=None):
    """Batched iLQR in float64 over ragged horizons: the clipped-Hessian backward pass, 16 step sizes at once."""
    B, n = x0.shape
    Tm, dev = int(T.max()), x0.device
    act = torch.arange(Tm, device=dev)[None, :] < T[:, None]
    alphas = DECAY ** torch.arange(N_ALPHA, dtype=torch.float64, device=dev)
    rows = torch.arange(B, device=dev)
    jac, hess, grad = torch.func.jacfwd, torch.func.hessian, torch.func.grad

    def rollout(U, X=None, K=None, k=None):
        """open loop (K None), or every step size's closed loop: X B x A x (Tm+1) x n, U, J B x A"""
        A = 1 if K is None else N_ALPHA
        x = x0[:, None].expand(B, A, n)
        xs, us, J = [x], [], torch.zeros(B, A, dtype=torch.float64, device=dev)
        for t in range(Tm):
            u = U[:, t][:, None].expand(B, A, m) if actor is None or K is not None else _actor(actor, x)
            if K is not None:
                u = u + alphas[None, :, None] * k[:, t][:, None] + torch.einsum("bmn,ban->bam", K[:, t], x - X[:, t][:, None])
            on = act[:, t][:, None]
            J = torch.where(on, J + sysm.l(x, u), J)
            x = torch.where(on[..., None], sysm.f(x, u), x)
            us.append(torch.where(on[..., None], u, torch.zeros_like(u)))
            xs.append(x)
        return torch.stack(xs, 2), torch.stack(us, 2), J + sysm.lT(x)

    def backward(X, U):
        x, u = X[:, :Tm].reshape(-1, n), U.reshape(-1, m)
        sh = lambda t: t.reshape(B, Tm, *t.shape[1:])  # noqa: E731
        fx, fu = _chunks(jac(sysm.f, (0, 1)), x, u)
        lx, lu = _chunks(grad(sysm.l, (0, 1)), x, u)
        lxx, luu = _chunks(lambda a, b: (hess(sysm.l, 0)(a, b), hess(sysm.l, 1)(a, b)), x, u)
        fx, fu, lx, lu, lxx, luu = (sh(t) for t in (fx, fu, lx, lu, _clip(lxx), _clip(luu)))
        xT = X[rows, T.long()]
        V, v = _clip(_chunks(hess(sysm.lT), xT)), _chunks(grad(sysm.lT), xT)
        K, k = torch.zeros(B, Tm, m, n, dtype=torch.float64, device=dev), torch.zeros(B, Tm, m, dtype=torch.float64, device=dev)
        Vx = torch.zeros(B, Tm + 1, n, dtype=torch.float64, device=dev)
        Vx[rows, T.long()] = v
        for t in range(Tm - 1, -1, -1):
            A, Bm, on = fx[:, t], fu[:, t], act[:, t]
            VA, VB = V @ A, V @ Bm
            Qxx, Qux, Quu = lxx[:, t] + A.mT @ VA, Bm.mT @ VA, luu[:, t] + Bm.mT @ VB
            Qx = lx[:, t] + torch.einsum("bij,bi->bj", A, v)
            Qu = lu[:, t] + torch.einsum("bij,bi->bj", Bm, v)
            G = -torch.linalg.solve(Quu, torch.cat([Qux, Qu[..., None]], -1))
            Kt, kt = G[..., :n], G[..., n]
            Vn = Qxx + Qux.mT @ Kt
            V = torch.where(on[:, None, None], 0.5 * (Vn + Vn.mT), V)
            v = torch.where(on[:, None], Qx + torch.einsum("bij,bi->bj", Qux, kt), v)
            K[:, t] = torch.where(on[:, None, None], Kt, K[:, t])
            k[:, t] = torch.where(on[:, None], kt, k[:, t])
            Vx[:, t] = torch.where(on[:, None], v, Vx[:, t])
        return K, k, Vx

    X, U, J = (t[:, 0] for t in rollout(torch.zeros(B, Tm, m, dtype=torch.float64, device=dev)))
    hist = [J]
    for _ in range(iters):
        K, k, _v = backward(X, U)
        Xc, Uc, Jc = rollout(U, X, K, k)
        better = Jc < J[:, None]
        if not bool(better.any(1).all()):
            return None                          # an instance stopped early: no fixed budget to compare
        j = better.int().argmax(1)
        X, U, J = Xc[rows, j], Uc[rows, j], Jc[rows, j]
        hist.append(J)
    out = {"J": J, "X": X, "U": U, "J_hist": torch.stack(hist, 1)}
    if vx:
        K, k, out["Vx"] = backward(X, U)
        out["K"] = K
    if window:
        lk = torch.cat([torch.where(act, sysm.l(X[:, :Tm], U), 0.0), torch.zeros(B, 1, dtype=torch.float64, device=dev)], 1)
        lk[rows, T.long()] = sysm.lT(X[rows, T.long()])
        w = torch.nn.functional.pad(lk, (0, window + 1)).unfold(1, window + 1, 1)[:, :Tm + 1].clone()
        last = torch.arange(Tm + 1, device=dev)[None, :] + window
        w[..., -1] = torch.where(last == T[:, None], w[..., -1], 0.0)
        out["Vbar"] = w.sum(-1)
    return out


def _pad(t, T_max, at):
    """the time axis to T_max + at: states (at = 1) repeat the last one, controls (at = 0) are 0"""
    more = T_max + at - t.shape[1]
    return torch.cat([t, t[:, -1:].expand(-1, more, *t.shape[2:])], 1) if at else torch.nn.functional.pad(t, [0, 0] * (t.dim() - 2) + [0, more])


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "rank":
        x, w = _candidates(case, seed)
        n, w, x = x.shape[1], torch.from_numpy(w).double().to(dev), torch.from_numpy(x).to(dev)
        W1, b1, W2, b2, W3, b3 = torch.split(w, [256 * n, 256, 256 * 256, 256, 256, 1])
        h = torch.tanh(x @ W1.reshape(256, n).T + b1)
        z = torch.tanh(h @ W2.reshape(256, 256).T + b2) @ W3 + b3
        return {"idx": None, "scores": torch.nn.functional.softplus(z, threshold=1e9)}
    if case["system"] in ("planar3", "arm7") and case["prec"] == "mixed":
        return None          # chaotic in float32
    prob, x0, T = _inputs(case, seed)
    sysm = {"pointmass": _PointMass, "dubins": _Dubins}.get(case["system"])
    sysm = sysm(prob.params) if sysm else _Tree(prob)
    r = _ilqr(sysm, torch.from_numpy(x0).to(dev), torch.from_numpy(T).to(dev), prob.m, case["iters"], case["vx"], case["window"],
              prob.actor_w)
    if r is None:
        return None
    T_max = case["T_hi"]
    out = {"J": r["J"], "X": _pad(r["X"], T_max, 1), "U": _pad(r["U"], T_max, 0)}
    if case["entry"] == "solver":
        out["J_hist"] = r["J_hist"]
    if case["vx"]:
        out["K"] = _pad(r["K"], T_max, 0)
        out["Vx"] = _pad(r["Vx"], T_max + 1, 0)
    if case["window"]:
        out["Vbar"] = torch.nn.functional.pad(r["Vbar"], [0, T_max + 1 - r["Vbar"].shape[1]])
    return out
