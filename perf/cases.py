"""Performance cases of the batched soft-contact rollout library.

The cases are what programs ask of the library through its Python entry
points (`rollout`, `rollout_host`, `rollout_grad`, `rollout_grad_params`,
`eval_rhs`, `eval_rhs_vjp`): single calls of a control loop, the batched
forward rollouts, rollouts with their discrete adjoint (plain and with the
contacts-from-distance right-hand side), the model-parameter gradient of
system identification, and the right-hand side with its vector-Jacobian
product.  Scenes and input distributions are those of
`paper_2506_14186_gb300.workloads`.  Horizons are those of one control window (at
most a quarter of a second).  Lanes per environment are left to the library, as
a program does that has not called the autotuner.

Adaptive steps through frictional contacts amplify a rounding difference until
a step decision differs (a 1e-14 change of the box's start moves some step
counts within 0.05 s), so `exact` gives trajectories only where two correct
programs agree: the fixed-step scheme, and the arm over short windows.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_14186_gb300 as dmx
from paper_2506_14186_gb300 import workloads as W

DEVICE = "cuda"
RTOL, ATOL, H0 = 1e-6, 1e-8, 1e-3


# --------------------------------------------------------------------------- the cases
def _case(name, op, model, B, T=0.0, NI=1, method="dopri5", cfd=False):
    return {"name": name, "op": op, "model": model, "B": B, "T": T, "NI": NI, "method": method, "cfd": cfd}


def listed():
    return [
        # one state of the robot's dynamics: a controller or an outer integrator that asks for v'
        _case("rhs_quadruped_1", "rhs", "quadruped", 1),
        # one plant stepped over a control period from host buffers (the simulator in the loop)
        _case("plant_quadruped_1", "host", "quadruped", 1, T=0.05),
        # a handful of pushed boxes: a small planner's candidates, fewer than the GPU has sub-partitions
        _case("push_box_37", "rollout", "box", 37, T=0.05),
        # the benchmark's batch of box pushes over one window
        _case("push_box_4096", "rollout", "box", 4096, T=0.2),
        # a large, odd batch of tosses with the other adaptive scheme: flight, then the impact
        _case("toss_tsit5_20001", "rollout", "toss", 20001, T=0.2, method="tsit5"),
        # sampling-based control of the arm: candidates of a window with piecewise-constant torques
        _case("arm_1000", "rollout", "chain_cube", 1000, T=0.2, NI=5),
        # legged locomotion: robots with uneven horizons, feet landing
        _case("walk_quadruped_3000", "rollout", "quadruped", 3000, T=0.2),
        # gradient-based control of the arm: taped rollout and discrete adjoint of a batch
        _case("grad_arm_2048", "grad", "chain_cube", 2048, T=0.2, NI=5),
        # trajectory optimisation of the robot through contacts from distance (straight-through)
        _case("grad_cfd_quadruped_300", "grad", "quadruped", 300, T=0.06, cfd=True),
        # gradients of the tosses with respect to their initial states
        _case("grad_toss_2048", "grad", "toss", 2048, T=0.25),
        # system identification: tosses with the gradient of every model parameter
        _case("params_toss_256", "params", "toss", 256, T=0.2),
        # linearisation at sampled states: vector-Jacobian products of the arm touching the cube
        _case("vjp_arm_16384", "vjp", "chain_cube", 16384),
    ]


# accepted steps per simulated second over these windows (start of the seeded trajectories)
STEPS_PER_S = {"ball": 60, "box": 1200, "toss": 320, "chain_cube": 300, "quadruped": 400, "arm_tilt": 500}


def _cost(c):
    """Right-hand-side equivalents of a case (a taped adjoint step counts four, with contacts from distance or
    the parameters twelve)."""
    if c["op"] in ("rhs", "vjp"):
        return c["B"] * (1 if c["op"] == "rhs" else 3)
    stages = 1 if c["method"] == "euler" else 6
    rate = 1.0 / H0 if c["method"] == "euler" else STEPS_PER_S[c["model"]]
    per = {"rollout": 1, "host": 1, "grad": 4, "params": 12}[c["op"]] * (3 if c["cfd"] else 1)
    size = {"ball": 0.5, "box": 1, "toss": 1, "chain_cube": 4, "arm_tilt": 5, "quadruped": 6}[c["model"]]
    return c["B"] * c["T"] * rate * stages * per * size


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        op = rng.choice(["rollout", "rollout", "rollout", "host", "grad", "grad", "params", "rhs", "vjp"])
        if op in ("rhs", "vjp"):
            model = rng.choice(["ball", "box", "chain_cube", "quadruped"])
            return {"op": op, "model": model, "B": log_int(1, 40000), "T": 0.0, "NI": 1, "method": "dopri5",
                    "cfd": rng.random() < 0.3}
        if op == "params":
            model = rng.choice(["toss", "ball"])
        else:
            model = rng.choice(["ball", "box", "toss", "chain_cube", "chain_cube", "quadruped", "quadruped"])
        method = rng.choice(["dopri5", "dopri5", "tsit5", "euler"])
        B = log_int(1, {"rollout": 20000, "host": 4096, "grad": 4096, "params": 400}[op])
        c = {"op": op, "model": model, "B": B, "T": round(rng.uniform(0.02, 0.25 if model in ("toss", "ball") else 0.2), 3),
             "NI": rng.randint(1, 5) if model == "chain_cube" else 1, "method": method,
             "cfd": op == "grad" and rng.random() < 0.3}
        # no costlier than the listed ones of its kind
        if _cost(c) <= {"rollout": 8e6, "host": 2e6, "grad": 3e6, "params": 1.2e6}[op]:
            return c


# --------------------------------------------------------------------------- inputs and calls
def _scene(case):
    opt = W.CFD_OPTIONS if case["cfd"] else {}
    return W.toss_scene() if case["model"] == "toss" and not opt else \
        W.box_scene(solref=(0.005, 1.0), **opt) if case["model"] == "toss" else W.SCENES[case["model"]](**opt)


def _inputs(case, seed):
    """Seeded initial states, horizons and controls of a rollout (host arrays, environment first)."""
    m, B, T = case["model"], case["B"], case["T"]
    if m == "quadruped":
        inp = W.quadruped_inputs(B, seed=seed)
        # released just above the ground, so that the feet land within the window; uneven horizons
        inp["x0"][:, 2] = 0.426 + np.random.default_rng(seed + 1).uniform(0.0, 0.004, B)
        inp["T"] = T * (0.25 + 0.75 * (inp["T"] - 0.5) / 2.5)
    elif m == "chain_cube":
        inp = W.chain_inputs(B, seed=seed, T=T, NI=case["NI"])
    else:
        inp = W.INPUTS[m](B, seed=seed, T=T)
        if m == "ball":   # drops that reach the ground within the window
            inp["x0"][:, 2] = 0.1 + np.random.default_rng(seed + 1).uniform(0.0, 0.1, B)
    return inp


def _states(case, seed):
    """Seeded states in contact: q [B, nq], v [B, nv], u [B, nu]."""
    g = np.random.default_rng(seed)
    m, B = case["model"], case["B"]
    sc = W.SCENES[m]()
    nq, nv, nu = W.scene_dims(sc)
    q = np.tile(np.asarray(sc["qpos0"]), (B, 1))
    v = g.normal(0.0, 0.3, (B, nv))
    u = g.normal(0.0, 0.3, (B, nu))

    def tilt(quat, s):
        d = np.concatenate([np.ones((B, 1)), g.normal(0.0, s, (B, 3))], axis=1)
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        w, x, y, z = quat.T
        a, b, c, e = d.T
        return np.stack([w * a - x * b - y * c - z * e, w * b + x * a + y * e - z * c,
                         w * c - x * e + y * a + z * b, w * e + x * c - y * b + z * a], axis=1)

    if m == "ball":
        q[:, 2] = 0.1 - g.uniform(-0.2e-3, 0.8e-3, B)
        q[:, 3:7] = tilt(q[:, 3:7], 0.5)
    elif m == "box":
        q[:, 2] = 0.05 - g.uniform(0.0, 1e-3, B)
        yaw = g.uniform(-math.pi, math.pi, B)
        q[:, 3:7] = tilt(np.stack([np.cos(yaw / 2), 0 * yaw, 0 * yaw, np.sin(yaw / 2)], axis=1), 0.003)
    elif m == "chain_cube":
        # the outstretched arm's last links pressed against the turned cube resting on the plane
        q[:, :7] = g.normal(0.0, 2e-3, (B, 7))
        yaw = g.uniform(0.05, 0.4, B) * g.choice([-1.0, 1.0], B)
        reach = 0.05 * (np.cos(yaw) + np.abs(np.sin(yaw)))
        q[:, 7] = 1.85 + g.uniform(-0.2, 0.1, B)
        q[:, 8] = 0.025 + reach - g.uniform(0.0, 2e-3, B)
        q[:, 9] = 0.05 - g.uniform(0.0, 5e-4, B)
        q[:, 10:14] = np.stack([np.cos(yaw / 2), 0 * yaw, 0 * yaw, np.sin(yaw / 2)], axis=1)
    else:
        q[:, 2] = 0.425 + g.uniform(-3e-3, 1e-3, B)
        q[:, 3:7] = tilt(q[:, 3:7], 0.003)
        q[:, 7:] = g.normal(0.0, 0.02, (B, nq - 7))
    return q, v, u


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEVICE)


def prepare(case, seed):
    s = {"op": case["op"], "cfd": case["cfd"], "model": dmx.Model(_scene(case))}
    if case["op"] in ("rhs", "vjp"):
        q, v, u = _states(case, seed)
        s["q"], s["v"], s["u"] = _dev(q.T), _dev(v.T), _dev(u.T) if u.shape[1] else None
        s["abar"] = _dev(np.random.default_rng(seed + 7).normal(size=v.shape).T)
        return s
    inp = _inputs(case, seed)
    ctrl = None if inp["ctrl"] is None else np.transpose(inp["ctrl"], (1, 2, 0))
    s["opts"] = {"NI": inp["NI"], "rtol": RTOL, "atol": ATOL, "h0": H0, "max_steps": 20000, "method": case["method"]}
    if case["op"] == "host":
        pin = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64).pin_memory()  # noqa: E731
        s["x0"], s["T"], s["ctrl"] = pin(inp["x0"].T), pin(inp["T"]), None if ctrl is None else pin(ctrl)
        return s
    s["x0"], s["T"], s["ctrl"] = _dev(inp["x0"].T), _dev(inp["T"]), None if ctrl is None else _dev(ctrl)
    if case["op"] in ("grad", "params"):
        s["opts"]["max_steps"] = 2000      # the tape holds every accepted step size
        s["xT_bar"] = _dev(np.random.default_rng(seed + 7).normal(size=inp["x0"].shape).T)
    return s


def run(s):
    m, op = s["model"], s["op"]
    if op == "rhs":
        a, info = dmx.eval_rhs(m, s["q"], s["v"], u=s["u"], cfd=s["cfd"])
        return {"a": a, "info": info}
    if op == "vjp":
        qb, vb, ub, st = dmx.eval_rhs_vjp(m, s["q"], s["v"], s["abar"], u=s["u"], cfd=s["cfd"])
        return {"qbar": qb, "vbar": vb, "ubar": ub, "status": st}
    if op == "host":
        return dmx.rollout_host(m, s["x0"], s["T"], ctrl=s["ctrl"], **s["opts"])
    if op == "rollout":
        out = dmx.rollout(m, s["x0"], s["T"], ctrl=s["ctrl"], **s["opts"])
        return {k: out[k] for k in ("xT", "nsteps", "nrej", "status")}
    out = dmx.rollout(m, s["x0"], s["T"], ctrl=s["ctrl"], tape=True, **s["opts"])
    res = {"xT": out["xT"], "nsteps": out["nsteps"], "status": out["status"]}
    if op == "grad":
        res["x0_bar"], res["ctrl_bar"] = dmx.rollout_grad(out["tape"], s["xT_bar"], cfd=s["cfd"])
    else:
        res["x0_bar"], res["ctrl_bar"], res["p_bar"], res["p_sum"] = dmx.rollout_grad_params(out["tape"], s["xT_bar"])
    return res


# FP64 operations of one right-hand side (box and arm: counted by the CPU oracle's counting scalar, the
# others in proportion to bodies, dofs and contact rows)
RHS_FLOPS = {"ball": 1500, "box": 4800, "toss": 4800, "chain_cube": 24700, "arm_tilt": 27000, "quadruped": 26000}


def work(case):
    nq, nv, nu = W.scene_dims(W.SCENES[case["model"]]())
    nx, B, f = nq + nv, case["B"], RHS_FLOPS[case["model"]]
    if case["op"] == "rhs":
        return {"bytes": B * (8 * (nx + nu + nv) + 16), "flops": B * f}
    if case["op"] == "vjp":
        return {"bytes": B * (8 * (2 * (nx + nu) + nv) + 4), "flops": B * 3 * f}
    rate = 1.0 / H0 if case["method"] == "euler" else STEPS_PER_S[case["model"]]
    steps = B * max(1.0, rate * case["T"] * (0.625 if case["model"] == "quadruped" else 1.0))
    stages = 1 if case["method"] == "euler" else 6
    bytes_ = B * 8 * (2 * nx + 1 + case["NI"] * nu)
    flops = steps * stages * f
    if case["op"] in ("grad", "params"):
        bytes_ += B * 8 * (2 * nx + case["NI"] * nu) + steps * 8
        flops *= 4 if case["op"] == "grad" else 12
    return {"bytes": bytes_, "flops": flops}


# --------------------------------------------------------------------------- 64-bit values in plain torch
# The same equations written with batched matrix algebra (body Jacobians, no spatial vectors): v' from
# M v' = tau - c + J^T f with the soft-contact forces at the minimum of the relaxed Gauss principle.
def _quat_mat(q):
    q = q / q.norm(dim=-1, keepdim=True)
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(*q.shape[:-1], 3, 3)


class _Reference:
    def __init__(self, scene, cfd=False):
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=DEVICE)  # noqa: E731
        self.bodies, o = scene["bodies"], scene["options"]
        self.nb = len(self.bodies)
        self.qa, self.va, self.parent, anc = [], [], [], []
        nq = nv = 0
        self.dof_body = []
        for b, d in enumerate(self.bodies):
            self.qa.append(nq)
            self.va.append(nv)
            free = d["joint"] == "free"
            self.dof_body += [b] * (6 if free else 1)
            nq, nv = nq + (7 if free else 1), nv + (6 if free else 1)
            anc.append({b} | (anc[d["parent"]] if d["parent"] >= 0 else set()))
        self.nq, self.nv = nq, nv
        self.mask = t([[1.0 if self.dof_body[i] in anc[b] else 0.0 for i in range(nv)] for b in range(self.nb)])
        self.lin = torch.zeros(nv, 3, dtype=torch.float64, device=DEVICE)
        for b, d in enumerate(self.bodies):
            if d["joint"] == "free":
                for k in range(3):
                    self.lin[self.va[b] + k, k] = 1.0
        self.damp = t([self.bodies[b]["damping"] for b in self.dof_body])
        self.mass, self.com = t([d["mass"] for d in self.bodies]), t([d["com"] for d in self.bodies])
        self.inertia = t([d["inertia"] for d in self.bodies])
        self.axis = [t(d["axis"]) / t(d["axis"]).norm() for d in self.bodies]
        self.pos, self.Roff = [t(d["pos"]) for d in self.bodies], [_quat_mat(t(d["quat"])) for d in self.bodies]
        self.grav = t(o["gravity"])
        self.acts = [(a["type"], self.qa[a["body"]], self.va[a["body"]], a["gear"], a["kp"], a["kd"])
                     for a in scene["actuators"]]
        tc, damp = o["solref"]
        dw = o["solimp"][1]
        self.b, self.k = 2.0 / (dw * tc), 1.0 / (dw * tc * damp) ** 2
        self.solimp, self.cfdimp, self.sp, self.cfd = o["solimp"], o["solimp_cfd"], o["softplus"], cfd
        self.thr = o["solimp_cfd"][2] if cfd else 0.0
        geoms = [(g["type"], g["body"], t(g["pos"]), _quat_mat(t(g["quat"])), g["size"]) for g in scene["geoms"]]
        invw = self._inverse_weights(t(scene["qpos0"]))
        self.plane, self.capbox = [], []     # (body, local point, radius, condim, mu, A_hat), capsule-box pairs
        for p in scene["pairs"]:
            ty, b, gp, gR, sz = geoms[p["geom1"]]
            if p["geom2"] < 0:
                local = {"sphere": [[0, 0, 0]], "capsule": [[-sz[1], 0, 0], [sz[1], 0, 0]],
                         "box": [[sz[0] if j & 1 else -sz[0], sz[1] if j & 2 else -sz[1], sz[2] if j & 4 else -sz[2]]
                                 for j in range(8)]}[ty]
                for x in local:
                    self.plane.append((b, gp + gR @ t([float(c) for c in x]), 0.0 if ty == "box" else sz[0],
                                       p["condim"], p["mu"], float(invw[b])))
            else:
                g2 = geoms[p["geom2"]]
                self.capbox.append((b, gp, gR[:, 0], sz[0], sz[1], g2[1], g2[2], g2[3], t(list(g2[4])), p["condim"],
                                    p["mu"], float(invw[b] + invw[g2[1]])))
        self.flat = [s for s in self.plane]
        if self.plane:
            self.pl_body = [s[0] for s in self.plane]
            self.pl_x = torch.stack([s[1] for s in self.plane])
            self.pl_r = t([s[2] for s in self.plane])
        dims = [(s[3], s[4], s[5]) for s in self.plane] + [(s[9], s[10], s[11]) for s in self.capbox]
        self.condim3 = bool(dims) and dims[0][0] == 3       # one contact dimension per scene here
        self.mu = t([d[1] for d in dims])
        self.ahat = t([d[2] * (1 + d[1] ** 2 if d[0] == 3 else 1.0) for d in dims])

    def _bodies(self, q):
        R, p = [], []
        for b, d in enumerate(self.bodies):
            x = q[:, self.qa[b]:]
            if d["joint"] == "free":
                R.append(_quat_mat(x[:, 3:7]))
                p.append(x[:, :3])
                continue
            a, th = self.axis[b], x[:, 0]
            K = torch.tensor([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]], dtype=torch.float64, device=DEVICE)
            Rj = torch.eye(3, dtype=torch.float64, device=DEVICE) + torch.sin(th)[:, None, None] * K \
                + (1 - torch.cos(th))[:, None, None] * (K @ K)
            Rl = self.Roff[b] @ Rj
            if d["parent"] < 0:
                R.append(Rl)
                p.append(self.pos[b].expand(q.shape[0], 3))
            else:
                Rp = R[d["parent"]]
                R.append(Rp @ Rl)
                p.append(p[d["parent"]] + Rp @ self.pos[b])
        W_ = []
        for b, d in enumerate(self.bodies):
            if d["joint"] == "free":
                W_ += [torch.zeros_like(p[b])] * 3 + [R[b][:, :, k] for k in range(3)]
            else:
                W_.append(R[b] @ self.axis[b])
        return torch.stack(R, 1), torch.stack(p, 1), torch.stack(W_, 1)

    def _point_jac(self, X, body, W_, O):
        """[B, n, nv, 3]: velocity of points X [B, n, 3] on `body` (list) per dof."""
        J = self.lin + torch.linalg.cross(W_[:, None], X[:, :, None] - O[:, None])
        return J * self.mask[body][None, :, :, None]

    def _mass(self, q):
        R, p, W_ = self._bodies(q)
        O = p[:, self.dof_body]
        X = p + torch.einsum("bnij,nj->bni", R, self.com)
        Jv = self._point_jac(X, list(range(self.nb)), W_, O)
        Jw = W_[:, None] * self.mask[None, :, :, None]
        I = torch.einsum("bnij,nj,bnkj->bnik", R, self.inertia, R)
        M = torch.einsum("n,bnid,bnjd->bij", self.mass, Jv, Jv) + torch.einsum("bnid,bnde,bnje->bij", Jw, I, Jw)
        return R, p, W_, O, X, Jv, Jw, I, M

    def _inverse_weights(self, q0):
        *_, Jv, Jw, I, M = self._mass(q0[None])
        Mi = torch.linalg.inv(M[0])
        return torch.einsum("nid,ij,njd->n", Jv[0], Mi, Jv[0]) / 3.0

    def _shape(self, x, mid, pw):
        if mid <= 0:
            return 1 - (1 - x) ** pw
        return torch.where(x <= mid, x ** pw / mid ** (pw - 1), 1 - (1 - x) ** pw / (1 - mid) ** (pw - 1) if mid < 1 else x ** pw)

    def _impedance(self, r):
        d0, dw, width, mid, pw = self.solimp
        d = d0 + (dw - d0) * self._shape((r.abs() / width).clamp(max=1.0), mid, pw)
        if self.cfd:
            dc, d1, wc, mc, pc = self.cfdimp
            d = torch.where(r >= 0, dc + (d1 - dc) * self._shape((1 - r / wc).clamp(0.0, 1.0), mc, pc), d)
        return d.clamp(0.0, 0.9999)

    @staticmethod
    def _box_distance(y, h):
        qd = y.abs() - h
        out = qd.clamp(min=0.0)
        inside = qd.max(-1).values
        is_out = inside > 0
        dist = torch.where(is_out, torch.where(is_out[..., None], out, torch.ones_like(out)).norm(dim=-1), inside)
        grad = torch.where(is_out[..., None], out / dist[..., None].abs().clamp(min=1e-300),
                           torch.nn.functional.one_hot(qd.argmax(-1), 3).to(y.dtype))
        return dist, grad * torch.where(y < 0, -1.0, 1.0)

    def _capsule_box(self, R, p, c):
        b1, gp, gu, rc, L, b2, gp2, gR2, h = c[:9]
        c1, u = p[:, b1] + R[:, b1] @ gp, R[:, b1] @ gu
        R2, c2 = R[:, b2] @ gR2, p[:, b2] + R[:, b2] @ gp2
        y0, w = torch.einsum("bji,bj->bi", R2, c1 - c2), torch.einsum("bji,bj->bi", R2, u)

        def slope(s):
            return (self._box_distance(y0 + s[:, None] * w, h)[1] * w).sum(-1)

        with torch.no_grad():
            lo, hi = torch.full_like(y0[:, 0], -L), torch.full_like(y0[:, 0], L)
            for _ in range(70):
                mid = 0.5 * (lo + hi)
                neg = slope(mid) < 0
                lo, hi = torch.where(neg, mid, lo), torch.where(neg, hi, mid)
            s = 0.5 * (lo + hi)
            y = y0 + s[:, None] * w
            dist, g = self._box_distance(y, h)
            on = (y.abs() > h).to(y.dtype)
            curv = ((w * w * on).sum(-1) - (g * w).sum(-1) ** 2) / dist
            free = (s > -L * (1 - 1e-12)) & (s < L * (1 - 1e-12)) & (dist > 0) & (curv > 1e-12)
            s = torch.where(s <= -L * (1 - 1e-12), -L, torch.where(s >= L * (1 - 1e-12), L, s))
        if torch.is_grad_enabled():   # the minimiser by the implicit function theorem
            sl = slope(s)
            s = s - torch.where(free, (sl - sl.detach()) / torch.where(free, curv, torch.ones_like(curv)), 0.0)
        dist, g = self._box_distance(y0 + s[:, None] * w, h)
        n = torch.einsum("bij,bj->bi", R2, g)
        r = dist - rc
        pos = c1 + s[:, None] * u - (rc + 0.5 * r)[:, None] * n
        ref = torch.where((n[:, 2:].abs() >= 0.5), torch.tensor([1.0, 0, 0], dtype=n.dtype, device=n.device),
                          torch.tensor([0, 0, 1.0], dtype=n.dtype, device=n.device))
        t1 = torch.linalg.cross(n, ref)
        t1 = t1 / t1.norm(dim=-1, keepdim=True)
        return r, pos, n, t1, torch.linalg.cross(n, t1)

    def rhs(self, q, v, u):
        R, p, W_, O, X, Jv, Jw, I, M = self._mass(q)
        B = q.shape[0]
        om = torch.einsum("bnid,bi->bnd", Jw, v)
        Xd = torch.einsum("bnid,bi->bnd", Jv, v)
        pd = torch.einsum("bnid,bi->bnd", self._point_jac(p, list(range(self.nb)), W_, O), v)
        Wd = torch.linalg.cross(om[:, self.dof_body], W_)
        al = torch.einsum("bid,ni,bi->bnd", Wd, self.mask, v)
        dJ = torch.linalg.cross(Wd[:, None], X[:, :, None] - O[:, None]) \
            + torch.linalg.cross(W_[:, None], Xd[:, :, None] - pd[:, self.dof_body][:, None])
        acc = torch.einsum("bnid,ni,bi->bnd", dJ, self.mask, v) - self.grav
        tq = torch.einsum("bnde,bne->bnd", I, al) + torch.linalg.cross(om, torch.einsum("bnde,bne->bnd", I, om))
        c = torch.einsum("n,bnid,bnd->bi", self.mass, Jv, acc) + torch.einsum("bnid,bnd->bi", Jw, tq)
        tau = -self.damp * v
        for a, (ty, qa, va, gear, kp, kd) in enumerate(self.acts):
            one = torch.zeros(self.nv, dtype=q.dtype, device=q.device)
            one[va] = 1.0
            f = gear * u[:, a] if ty == "motor" else kp * (u[:, a] - q[:, qa]) - kd * v[:, va]
            tau = tau + f[:, None] * one
        rhs0 = tau - c
        r, Js = [], []
        if self.plane:
            pt = p[:, self.pl_body] + torch.einsum("bnij,nj->bni", R[:, self.pl_body], self.pl_x)
            rp = pt[..., 2] - self.pl_r
            pos = torch.cat([pt[..., :2], (pt[..., 2] - (self.pl_r + 0.5 * rp))[..., None]], -1)
            r.append(rp)
            Jp = self._point_jac(pos, self.pl_body, W_, O)
            Js.append(torch.stack([Jp[..., 2], Jp[..., 0], Jp[..., 1]], 2))
        for cb in self.capbox:
            rc, pos, n, t1, t2 = self._capsule_box(R, p, cb)
            Jp = (self._point_jac(pos[:, None], [cb[0]], W_, O) - self._point_jac(pos[:, None], [cb[5]], W_, O))[:, 0]
            r.append(rc[:, None])
            Js.append(torch.stack([(Jp * e[:, None]).sum(-1) for e in (n, t1, t2)], 1)[:, None])
        r, Js = torch.cat(r, 1), torch.cat(Js, 1)         # [B, ns], [B, ns, 3, nv]
        inc = r < self.thr
        d = self._impedance(r)
        pterm = self.k * d * self.sp * torch.nn.functional.softplus(-r / self.sp, threshold=1e9) if self.cfd else -self.k * d * r
        D = torch.where(inc, d / (self.ahat * (1 - d)), 0.0)
        if self.condim3:
            f1, f2 = self.mu[:, None] * Js[:, :, 1], self.mu[:, None] * Js[:, :, 2]
            J = torch.stack([Js[:, :, 0] + f1, Js[:, :, 0] - f1, Js[:, :, 0] + f2, Js[:, :, 0] - f2], 2).reshape(B, -1, self.nv)
            D, pterm = D.repeat_interleave(4, 1), pterm.repeat_interleave(4, 1)
        else:
            J = Js[:, :, 0]
        aref = -self.b * torch.einsum("bri,bi->br", J, v) + pterm
        return self._solve(M, rhs0, J, D, aref)

    def _solve(self, M, rhs0, J, D, aref):
        def target(act):
            w = torch.where(act, D, 0.0)
            H = M + torch.einsum("br,bri,brj->bij", w, J, J)
            L = torch.linalg.cholesky(H)
            return torch.cholesky_solve((rhs0 + torch.einsum("br,bri->bi", w * aref, J))[..., None], L)[..., 0]

        with torch.no_grad():
            a = target(torch.zeros_like(D, dtype=torch.bool))
            a0 = a
            res = lambda x: torch.einsum("bri,bi->br", J, x) - aref  # noqa: E731
            al = torch.tensor([0.5 ** k for k in range(14)], dtype=M.dtype, device=M.device)
            for _ in range(60):
                act = res(a) < 0
                an = target(act)
                if bool((((res(an) < 0) == act) | (D == 0)).all()):
                    break
                cand = a[:, None] + al[None, :, None] * (an - a)[:, None]
                e = cand - a0[:, None]
                z = (torch.einsum("bri,bki->bkr", J, cand) - aref[:, None]).clamp(max=0.0)
                cost = 0.5 * torch.einsum("bki,bij,bkj->bk", e, M, e) + 0.5 * (D[:, None] * z * z).sum(-1)
                best = cost.argmin(1)
                done = (((res(an) < 0) == act) | (D == 0)).all(1)
                a = torch.where(done[:, None], an, cand[torch.arange(len(a)), best])
        return target(act)

    def plus(self, q, dq):
        out = []
        for b, d in enumerate(self.bodies):
            qa, va = self.qa[b], self.va[b]
            if d["joint"] != "free":
                out.append(q[:, qa:qa + 1] + dq[:, va:va + 1])
                continue
            out.append(q[:, qa:qa + 3] + dq[:, va:va + 3])
            w = dq[:, va + 3:va + 6]
            th2 = (w * w).sum(-1, keepdim=True)
            th = th2.clamp(min=1e-24).sqrt()
            small = th2 < 1e-4
            cw = torch.where(small, 1 - th2 / 8 + th2 ** 2 / 384 - th2 ** 3 / 46080, torch.cos(0.5 * th))
            sk = torch.where(small, 0.5 - th2 / 48 + th2 ** 2 / 3840 - th2 ** 3 / 645120, torch.sin(0.5 * th) / th)
            e, x = sk * w, q[:, qa + 3:qa + 7]
            r = torch.cat([x[:, :1] * cw - (x[:, 1:] * e).sum(-1, keepdim=True),
                           x[:, :1] * e + cw * x[:, 1:] + torch.linalg.cross(x[:, 1:], e)], -1)
            out.append(r / r.norm(dim=-1, keepdim=True))
        return torch.cat(out, 1)

    def magnitude(self, q):
        cols = []
        for b, d in enumerate(self.bodies):
            if d["joint"] == "free":
                cols += [q[:, self.qa[b]:self.qa[b] + 3].abs(), torch.ones_like(q[:, :3])]
            else:
                cols.append(q[:, self.qa[b]:self.qa[b] + 1].abs())
        return torch.cat(cols, 1)


def _tableau(method):
    if method == "dopri5":
        a = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
             [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
             [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
             [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]]
        bh = [5179 / 57600, 0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40]
        return a, [x - y for x, y in zip(a[6] + [0.0], bh)]
    a = [[], [0.161], [-0.008480655492356989, 0.335480655492357],
         [2.897153057105493, -6.359448489975075, 4.3622954328695815],
         [5.325864828439257, -11.748883564062828, 7.4955393428898365, -0.09249506636175525],
         [5.86145544294642, -12.92096931784711, 8.159367898576159, -0.071584973281401, -0.028269050394068383],
         [0.09646076681806523, 0.01, 0.4798896504144996, 1.379008574103742, -3.290069515436081, 2.324710524099774]]
    return a, [-0.00178001105222577714, -0.0008164344596567469, 0.007880878010261995, -0.1447110071732629,
               0.5823571654525552, -0.45808210592918697, 0.015151515151515152]


def _step(ref, method, q, v, u, h):
    """One step of the scheme: new state and the RMS error terms (None for the fixed step)."""
    h = h[:, None]
    if method == "euler":
        vn = v + h * ref.rhs(q, v, u)
        return ref.plus(q, h * vn), vn, None
    a, e = _tableau(method)
    V, K = [v], [ref.rhs(q, v, u)]
    qs, vs = q, v
    for s in range(1, 7):
        vs = v + h * sum(c * k for c, k in zip(a[s], K) if c)
        qs = ref.plus(q, h * sum(c * x for c, x in zip(a[s], V) if c))
        V.append(vs)
        K.append(ref.rhs(qs, vs, u))
    ep, ev = (h * sum(c * x for c, x in zip(e, L) if c) for L in (V, K))
    rp = ep / (ATOL + RTOL * torch.maximum(ref.magnitude(q), ref.magnitude(qs)))
    rv = ev / (ATOL + RTOL * torch.maximum(v.abs(), vs.abs()))
    return qs, vs, ((rp * rp + rv * rv).sum(1) / (2 * ref.nv)).sqrt()


def _exact_rollout(case, seed):
    ref, inp = _Reference(_scene(case)), _inputs(case, seed)
    x0, T, NI, method = _dev(inp["x0"]), _dev(inp["T"]), inp["NI"], case["method"]
    q, v = x0[:, :ref.nq].clone(), x0[:, ref.nq:].clone()
    ctrl = None if inp["ctrl"] is None else _dev(inp["ctrl"])
    B = q.shape[0]
    t, h, lp = torch.zeros_like(T), torch.full_like(T, H0), torch.zeros_like(T)
    k = torch.zeros(B, dtype=torch.long, device=DEVICE)
    log = []
    while bool((t < T).any()) and len(log) < 1500:
        live = t < T
        ku = k.clamp(max=NI - 1)
        tn = torch.where(k + 1 >= NI, T, T * (k + 1) / NI)
        hb = tn - t
        clamp = (h >= hb) | (hb - h < 1e-12)
        ht = torch.where(live, torch.where(clamp, hb, h), torch.zeros_like(h))
        u = None if ctrl is None else ctrl[torch.arange(B), ku]
        qs, vs, err = _step(ref, method, q, v, u, ht)
        ok = live if err is None else live & (err <= 1.0)
        log.append((q, v, ht, ku, ok))
        reached = ok & (clamp | (t + ht >= tn))
        t = torch.where(reached, tn, torch.where(ok, t + ht, t))
        k = torch.where(reached, k + 1, k)
        q, v = torch.where(ok[:, None], qs, q), torch.where(ok[:, None], vs, v)
        if err is None:
            h = torch.full_like(h, H0)
            continue
        le = err.clamp(min=1e-10).log()
        grow = (0.9 * torch.exp(-0.12 * le + 0.04 * lp)).clamp(0.2, 10.0)
        cut = torch.nan_to_num(0.9 * err.clamp(min=1e-10) ** -0.2, nan=0.2).clamp(min=0.2)
        h = torch.where(ok, ht * grow, torch.where(live, ht * cut, h))
        lp = torch.where(ok, le, lp)
    return ref, ctrl, q, v, log


def _exact_grad(case, seed):
    ref, ctrl, q, v, log = _exact_rollout(case, seed)
    xT = torch.cat([q, v], 1)
    bar = _dev(np.random.default_rng(seed + 7).normal(size=tuple(xT.shape)))
    back = _Reference(_scene(case), cfd=case["cfd"]) if case["cfd"] else ref
    if case["cfd"]:
        return xT, None, None
    cb = None if ctrl is None else torch.zeros_like(ctrl)
    for q0, v0, h, ku, ok in reversed(log):
        x = torch.cat([q0, v0], 1).requires_grad_()
        u = None if ctrl is None else ctrl[torch.arange(len(ku)), ku].requires_grad_()
        qs, vs, _ = _step(back, case["method"], x[:, :ref.nq], x[:, ref.nq:], u, h)
        g = torch.autograd.grad(torch.cat([qs, vs], 1), [x] + ([] if u is None else [u]), bar)
        bar = torch.where(ok[:, None], g[0], bar)
        if u is not None:
            cb[torch.arange(len(ku)), ku] += torch.where(ok[:, None], g[1], torch.zeros_like(g[1]))
    return xT, bar, cb


def exact(case, seed):
    op = case["op"]
    if op in ("rhs", "vjp"):
        ref = _Reference(_scene(case), cfd=case["cfd"])
        q, v, u = (_dev(x) for x in _states(case, seed))
        if op == "rhs":
            return {"a": ref.rhs(q, v, u).T.contiguous(), "info": None}
        ab = _dev(np.random.default_rng(seed + 7).normal(size=tuple(v.shape)))
        x = [q.requires_grad_(), v.requires_grad_(), u.requires_grad_()]
        g = torch.autograd.grad(ref.rhs(*x), x, ab, allow_unused=True)
        return {"qbar": g[0].T.contiguous(), "vbar": g[1].T.contiguous(),
                "ubar": g[2].T.contiguous() if u.shape[1] else None, "status": None}
    # trajectories: where two programs agree (see above) and the torch program takes seconds
    T, euler, model = case["T"], case["method"] == "euler", case["model"]
    if not (euler and (model != "box" or T <= 0.05)) and not (model == "chain_cube" and T <= 0.1):
        return None
    calls = (T / H0 if euler else 6 * 500 * T) * (3 if model in ("chain_cube", "quadruped") else 1)
    if calls * (4 if op == "grad" and not case["cfd"] else 1) > 2500:
        return None
    if op == "grad":
        xT, xb, cb = _exact_grad(case, seed)
        return {"xT": xT.T.contiguous(), "nsteps": None, "status": None,
                "x0_bar": None if xb is None else xb.T.contiguous(),
                "ctrl_bar": None if cb is None else cb.permute(1, 2, 0).contiguous()}
    _, _, q, v, _ = _exact_rollout(case, seed)
    return {"xT": torch.cat([q, v], 1).T.contiguous()}
