"""The work that users of the simulator have it do, as cases to time.

A case is one call sequence through the public binding: a control-loop step, a
rollout with its gradients (terminal or per-step objectives), or a forward-mode
step derivative, over the model families of ``workloads`` (double pendulum,
serial chains, uneven trees, quadrupeds with and without foot contacts,
humanoids), their precisions and batch sizes.  Horizons are short enough that
rounding is not amplified by the systems' own (chaotic) sensitivity; the cost per
step does not depend on the horizon.

``exact`` states the same step independently in 64 bits: spatial quantities at
the world origin, links processed level by level over the whole batch, the
gradient as  -d(lambda . inverse dynamics)  with M lambda = d(objective)/d(qdd).
"""
import math

import numpy as np
import torch

import workloads as wl
from paper_2109_07719_gb300 import Rollout, RolloutTrajectory, Simulator

FAMILIES = ("pendulum", "chains", "trees", "quadruped", "humanoid", "quadruped_contact")


def _case(kind, family, precision, B, T=1, **more):
    c = {"kind": kind, "family": family, "precision": precision, "B": B, "T": T, "k": 1, "links": 0, "damping": False}
    c.update(more)
    return c


def listed():
    return [
        # a real-time control loop: one step of a few arms per tick, where latency and launches count
        dict(_case("step", "chains", "fp32", 64, links=7), name="step_chains_64"),
        # one double pendulum over 1000 steps with its gradient in FP64: the smallest system, pure latency
        dict(_case("rollout", "pendulum", "fp64", 1, T=1000), name="pendulum_fp64"),
        # trajectory optimisation / system identification on 7-DOF arms: gradients for torques and masses
        dict(_case("rollout", "chains", "fp32", 4096, T=128, links=7), name="chains_fp32"),
        # the same in FP64, a ragged batch
        dict(_case("rollout", "chains", "fp64", 1000, T=50, links=7), name="chains_fp64"),
        # the benchmark's mixed batch: trees of 2..64 links, laid out by link count
        dict(_case("rollout", "trees", "fp32", 16384, T=24, links=64), name="trees_fp32"),
        # long horizons on little memory: checkpoints every 8 steps, segments replayed; damped joints
        dict(_case("rollout", "trees", "fp32", 1500, T=48, k=8, links=40, damping=True), name="trees_replay"),
        # legged robots in the mixed mode (FP64 D-solves)
        dict(_case("rollout", "quadruped", "fp32_d64", 8192, T=60), name="quadrupeds_d64"),
        # per-step objectives (tracking costs) on humanoids
        dict(_case("trajectory", "humanoid", "fp32", 1024, T=60), name="humanoids_trajectory"),
        # quadrupeds landing on their feet: gradients through the contact solver
        dict(_case("rollout", "quadruped_contact", "fp64", 512, T=12), name="contacts_fp64"),
        # one-step Jacobian-vector products for sample enhancement
        dict(_case("jvp", "quadruped", "fp32", 4096), name="jvp_quadrupeds"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "rollout", "rollout", "rollout", "trajectory", "jvp"))
    family = rng.choice(("pendulum", "chains", "chains", "trees", "trees", "quadruped", "humanoid"))
    if kind == "rollout" and rng.random() < 0.15:
        family = "quadruped_contact"
    precision = rng.choice(("fp64", "fp32", "fp32", "fp32_d64"))
    if family == "quadruped_contact":
        return _case(kind, family, "fp64", _log(rng, 3, 600), T=rng.randint(2, 12))
    links = {"chains": rng.randint(2, 16), "trees": rng.randint(8, 64)}.get(family, 0)
    size = {"pendulum": 2, "chains": links, "trees": links / 2, "quadruped": 13, "humanoid": 23}[family]
    cap = 16000 * 7 / size * (0.2 if precision == "fp64" else 1.0)
    B = _log(rng, 1, min(16384, cap))
    T = 1 if kind in ("step", "jvp") else _log(rng, 4, 100)
    k = 1 if kind in ("step", "jvp") or rng.random() < 0.6 else rng.randint(2, min(T, 20))
    return _case(kind, family, precision, B, T=T, k=k, links=links,
                 damping=family in ("chains", "trees") and rng.random() < 0.3)


def _work_of(case, seed):
    """The workload's model and host initial state for these inputs."""
    f, kw = case["family"], dict(B=case["B"], T=case["T"], seed=wl.SEED_BASE + 17 * seed)
    if f == "pendulum":
        w = wl.double_pendulum(**kw)
    elif f == "chains":
        w = wl.serial_chains(n=case["links"], precision=case["precision"], **kw)
    elif f == "trees":
        # the trees' shapes go by the case alone, so that every seed has outputs of the same shape
        kw["seed"] = wl.SEED_BASE + case["links"]
        w = wl.uneven_trees(dof_lo=2, dof_hi=case["links"], precision=case["precision"], **kw).in_slot_order()
        w.q0 = np.ascontiguousarray(w.q0 * np.random.default_rng(seed).choice([-1.0, 1.0], w.q0.shape))
    elif f == "humanoid":
        w = wl.humanoid(precision=case["precision"], **kw)
    else:
        w = wl.quadruped(precision=case["precision"], contacts=f == "quadruped_contact", **kw)
    if case["damping"]:
        w.model = w.model.with_damping(seed + 3)
    return w


def _inputs(case, seed, w, device):
    """State, torques, tangents and objective gradients, float64 on `device`, rounded to the case's type."""
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    g = torch.Generator(device=device)
    g.manual_seed(1000003 * (seed + 1))
    m, B, T = w.model, case["B"], case["T"]
    nq, nv = m.nq_max, m.nv_max
    maskq = torch.as_tensor(np.arange(nq)[:, None] < m.nq_per_system()[None, :], device=device)
    maskv = torch.as_tensor(np.arange(nv)[:, None] < m.nv_per_system()[None, :], device=device)
    actuated = torch.as_tensor(w.tau_mask, device=device)

    def normal(*shape):
        return torch.randn(shape, generator=g, device=device, dtype=torch.float64)

    q0 = torch.tensor(w.q0, device=device)
    qd0 = 0.3 * normal(nv, B) * maskv
    if case["family"] == "quadruped_contact":  # straight legs, feet 1..4 mm into the ground, falling
        q0[7:] = 0.02 * normal(nq - 7, B)
        q0[2] = 0.42 - 0.001 - 0.003 * torch.rand(B, generator=g, device=device, dtype=torch.float64)
        qd0[3:6] = 0.0
        qd0[5] = -1.0
    d = {"q0": q0, "qd0": qd0, "tau": normal(T, nv, B) * w.tau_sigma * actuated,
         "mass": torch.as_tensor(m.mass, device=device) * (1.0 + 0.05 * torch.tanh(normal(m.n_links_total)))}
    if case["kind"] == "rollout":
        d["gq"], d["gqd"] = normal(nq, B) * maskq, normal(nv, B) * maskv
    elif case["kind"] == "trajectory":
        d["gx"] = normal(T + 1, nq + nv, B) * torch.cat([maskq, maskv])
    elif case["kind"] == "jvp":
        d["dq"], d["dqd"], d["dtau"] = normal(nq, B) * maskq, normal(nv, B) * maskv, normal(nv, B) * maskv
    return {n: x.to(dt) for n, x in d.items()}


def prepare(case, seed):
    w = _work_of(case, seed)
    sim = Simulator(w.model, precision=case["precision"])
    s = _inputs(case, seed, w, sim.device)
    if case["kind"] in ("rollout", "trajectory"):
        for n in ("q0", "qd0", "tau", "mass"):
            s[n].requires_grad_(True)
    else:
        s["tau"] = s["tau"][0].contiguous()
    return {"case": case, "sim": sim, **s}


def run(state):
    case, sim = state["case"], state["sim"]
    if case["kind"] == "step":
        q, qd = sim.step(state["q0"], state["qd0"], state["tau"])
        return {"q": q, "qd": qd}
    if case["kind"] == "jvp":
        out = sim.jvp(state["q0"], state["qd0"], state["tau"], state["dq"], state["dqd"], state["dtau"])
        return dict(zip(("q", "qd", "dq", "dqd"), out))
    x = [state[n] for n in ("q0", "qd0", "tau", "mass")]
    if case["kind"] == "trajectory":
        traj = RolloutTrajectory.apply(sim, *x, case["k"])
        g = torch.autograd.grad([traj], x, [state["gx"]])
        out = {"traj": traj.detach()}
    else:
        qT, qdT = Rollout.apply(sim, *x, case["k"])
        g = torch.autograd.grad([qT, qdT], x, [state["gq"], state["gqd"]])
        out = {"qT": qT.detach(), "qdT": qdT.detach()}
    out.update(zip(("gq0", "gqd0", "gtau", "gmass"), g))
    return out


def work(case):
    """Inputs read once and outputs written once; about 600 operations per link for a
    forward step and as many again for its adjoint after one recompute."""
    word = 8 if case["precision"] == "fp64" else 4
    B, T = case["B"], case["T"]
    links = {"pendulum": 2, "chains": case["links"], "trees": (2 + case["links"]) / 2, "humanoid": 23}.get(case["family"], 13)
    nq, nv = {"humanoid": (29, 28), "quadruped": (19, 18), "quadruped_contact": (19, 18)}.get(case["family"], (links, links))
    model, x = 23 * links, nq + nv
    if case["kind"] == "step":
        return {"bytes": B * word * (model + 2 * x + nv), "flops": B * 600 * links}
    if case["kind"] == "jvp":
        return {"bytes": B * word * (model + 4 * x + 2 * nv), "flops": B * 1800 * links}
    seeds = (T + 1) * x if case["kind"] == "trajectory" else x
    states = (T + 1) * x if case["kind"] == "trajectory" else x
    return {"bytes": B * word * (model + 2 * x + 2 * T * nv + seeds + states + links), "flops": B * T * 1800 * links}


# ------------------------------------------------------------------ the same step in 64 bits


def _skew(v):
    z = torch.zeros_like(v[..., 0])
    return torch.stack([z, -v[..., 2], v[..., 1], v[..., 2], z, -v[..., 0], -v[..., 1], v[..., 0], z], -1).reshape(v.shape[:-1] + (3, 3))


def _mv(M, v):
    return (M @ v[..., None])[..., 0]


def _quat_R(q):
    x, y, z, w = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1).reshape(q.shape[:-1] + (3, 3))


class _Plain:
    """A batch of trees, links grouped by depth.  Spatial vectors (angular, linear) at the world origin."""

    def __init__(self, m, dev):
        t = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
        B, off = m.n_systems, np.asarray(m.sys_link_offset)
        sysof = np.repeat(np.arange(B), np.diff(off))
        par = np.where(m.parent >= 0, m.parent + off[sysof], -1)
        depth = np.zeros(len(par), int)
        for i in range(int(np.diff(off).max())):  # parents precede children inside a system
            at = off[:-1][np.diff(off) > i] + i
            depth[at] = np.where(par[at] >= 0, depth[par[at]] + 1, 0)
        free = np.asarray(m.joint_type) == wl.FREE
        voff = np.zeros(len(par), int)
        nv, nq = np.where(free, 6, 1), np.where(free, 7, 1)
        voff, qoff = (np.cumsum(n) - n for n in (nv, nq))
        voff, qoff = (o - o[off[:-1]][sysof] for o in (voff, qoff))
        pos = np.zeros(len(par), int)
        self.levels = []
        for d in range(depth.max() + 1):
            at = np.nonzero(depth == d)[0]
            pos[at] = np.arange(len(at))
            ix = lambda a: torch.as_tensor(a, device=dev)  # noqa: E731
            self.levels.append({"at": ix(at), "sys": ix(sysof[at]), "v": ix(voff[at]), "q": ix(qoff[at]),
                                "par": ix(pos[par[at]]) if d else None, "free": bool(free[at].all())})
        self.B, self.dt, self.grav = B, m.dt, t(m.gravity)
        X = t(m.X_tree)
        self.E, self.r, self.axis, self.com = X[:, :9].reshape(-1, 3, 3), X[:, 9:], t(m.axis), t(m.com)
        ic = t(m.I_com)
        self.Ic = ic[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].reshape(-1, 3, 3)
        self.damp = t(m.damping) if m.damping is not None else torch.zeros(len(par), device=dev, dtype=torch.float64)
        self.dev = dev

    def geometry(self, q, mass):
        """Per level: motion subspace S [n, 6, dofs], spatial inertia [n, 6, 6]."""
        out, R, p = [], None, None
        for lv in self.levels:
            at, sy = lv["at"], lv["sys"]
            Et, rt = self.E[at].transpose(-1, -2), self.r[at]
            if lv["par"] is not None:
                Rp, pp = R[lv["par"]], p[lv["par"]]
                R0, p0 = Rp @ Et, pp + _mv(Rp, rt)
            else:
                R0, p0 = Et, rt
            if lv["free"]:
                Q = torch.stack([q[lv["q"] + i, sy] for i in range(7)], -1)
                p = p0 + _mv(R0, Q[:, :3])
                R = R0 @ _quat_R(Q[:, 3:])
                Z = torch.zeros_like(R)
                S = torch.cat([torch.cat([R, Z], -1), torch.cat([_skew(p) @ R, R], -1)], -2)
            else:
                a = self.axis[at]
                th = q[lv["q"], sy]
                K = _skew(a)
                J = torch.eye(3, device=self.dev, dtype=torch.float64) + torch.sin(th)[:, None, None] * K + \
                    (1 - torch.cos(th))[:, None, None] * (K @ K)
                p, R = p0, R0 @ J
                s = _mv(R, a)
                S = torch.cat([s, torch.linalg.cross(p, s)], -1)[..., None]
            c = p + _mv(R, self.com[at])
            m1, C = mass[at][:, None, None], _skew(c)
            eye = torch.eye(3, device=self.dev, dtype=torch.float64).expand_as(C)
            Iw = R @ self.Ic[at] @ R.transpose(-1, -2) - m1 * (C @ C)
            out.append((S, torch.cat([torch.cat([Iw, m1 * C], -1), torch.cat([-m1 * C, m1 * eye], -1)], -2)))
        return out

    def dofs(self, lv, x):
        n = 6 if lv["free"] else 1
        return torch.stack([x[lv["v"] + i, lv["sys"]] for i in range(n)], -1)

    def scatter(self, vals, nv):
        x = torch.zeros(nv, self.B, device=self.dev, dtype=torch.float64)
        for lv, y in zip(self.levels, vals):
            for i in range(y.shape[-1]):
                x = x.index_put((lv["v"] + i, lv["sys"]), y[:, i])
        return x

    @staticmethod
    def crf(v, f):
        w, u = v[..., :3], v[..., 3:]
        return torch.cat([torch.linalg.cross(w, f[..., :3]) + torch.linalg.cross(u, f[..., 3:]), torch.linalg.cross(w, f[..., 3:])], -1)

    @staticmethod
    def crm(v, m):
        w, u = v[..., :3], v[..., 3:]
        return torch.cat([torch.linalg.cross(w, m[..., :3]), torch.linalg.cross(w, m[..., 3:]) + torch.linalg.cross(u, m[..., :3])], -1)

    def inverse_dynamics(self, geo, qd, qdd):
        """Joint forces [per level] that give qdd (qdd None: zero), damping included."""
        v = a = None
        fs = []
        for lv, (S, I) in zip(self.levels, geo):
            x = self.dofs(lv, qd)
            vj = _mv(S, x)
            aj = _mv(S, self.dofs(lv, qdd)) if qdd is not None else 0.0
            if lv["par"] is None:
                v, a = vj, aj + torch.cat([torch.zeros(3, device=self.dev, dtype=torch.float64), -self.grav]).expand_as(vj)
            else:
                v = v[lv["par"]] + vj
                a = a[lv["par"]] + aj + self.crm(v, vj)
            fs.append(_mv(I, a) + self.crf(v, _mv(I, v)))
        out = []
        for d in range(len(fs) - 1, -1, -1):
            lv = self.levels[d]
            t = _mv(geo[d][0].transpose(-1, -2), fs[d])
            if not lv["free"]:
                t = t + self.damp[lv["at"]][:, None] * self.dofs(lv, qd)
            out.append(t)
            if lv["par"] is not None:
                fs[d - 1] = fs[d - 1].index_add(0, lv["par"], fs[d])
        return out[::-1]

    def factor(self, geo):
        """Articulated inertias: per level (U, D^-1)."""
        IA = [I for _, I in geo]
        out = [None] * len(geo)
        for d in range(len(geo) - 1, -1, -1):
            S = geo[d][0]
            U = IA[d] @ S
            Di = torch.linalg.inv(S.transpose(-1, -2) @ U) if S.shape[-1] > 1 else 1.0 / (S.transpose(-1, -2) @ U)
            out[d] = (U, Di)
            if d:
                IA[d - 1] = IA[d - 1].index_add(0, self.levels[d]["par"], IA[d] - U @ Di @ U.transpose(-1, -2))
        return out

    def solve(self, geo, fac, f):
        """M^-1 f, per level."""
        p = [torch.zeros(S.shape[0], 6, device=self.dev, dtype=torch.float64) for S, _ in geo]
        u = [None] * len(geo)
        for d in range(len(geo) - 1, -1, -1):
            S, (U, Di) = geo[d][0], fac[d]
            u[d] = f[d] - _mv(S.transpose(-1, -2), p[d])
            if d:
                p[d - 1] = p[d - 1].index_add(0, self.levels[d]["par"], p[d] + _mv(U @ Di, u[d]))
        a, x = None, []
        for d, (S, _) in enumerate(geo):
            U, Di = fac[d]
            ap = a[self.levels[d]["par"]] if d else torch.zeros_like(p[0])
            y = _mv(Di, u[d] - _mv(U.transpose(-1, -2), ap))
            a = ap + _mv(S, y)
            x.append(y)
        return x

    def accel(self, q, qd, tau, mass):
        geo = self.geometry(q, mass)
        bias = self.inverse_dynamics(geo, qd, None)
        fac = self.factor(geo)
        qdd = self.solve(geo, fac, [self.dofs(lv, tau) - b for lv, b in zip(self.levels, bias)])
        return geo, fac, self.scatter(qdd, qd.shape[0])

    def integrate(self, q, qd, qdd):
        v = qd + self.dt * qdd
        if not self.levels[0]["free"]:
            return q + self.dt * v, v
        Q, w, u = q[3:7].T, v[:3].T, v[3:6].T
        p = q[:3].T + self.dt * _mv(_quat_R(Q), u)
        x, y, z, s = Q.unbind(-1)
        a, b, c = w.unbind(-1)
        r = torch.stack([s * a + y * c - z * b, s * b + z * a - x * c, s * c + x * b - y * a, -x * a - y * b - z * c], -1)
        n = Q + 0.5 * self.dt * r
        n = n / n.norm(dim=-1, keepdim=True)
        return torch.cat([p.T, n.T, q[7:] + self.dt * v[6:]]), v

    def step(self, q, qd, tau, mass):
        return self.integrate(q, qd, self.accel(q, qd, tau, mass)[2])

    def pull_back(self, q, qd, tau, mass, gq, gqd):
        """Gradients of (gq . q', gqd . qd') for q, qd, tau, mass."""
        geo, fac, qdd = self.accel(q, qd, tau, mass)
        with torch.enable_grad():
            x = [y.detach().requires_grad_(True) for y in (q, qd, qdd)]
            bq, bqd, bqdd = torch.autograd.grad(self.integrate(*x), x, [gq, gqd])
            lam = [y.detach() for y in self.solve(geo, fac, [self.dofs(lv, bqdd) for lv in self.levels])]
            x = [y.detach().requires_grad_(True) for y in (q, qd, mass)]
            forces = self.inverse_dynamics(self.geometry(x[0], x[2]), x[1], qdd)
            g = torch.autograd.grad(sum((a * b).sum() for a, b in zip(forces, lam)), x, allow_unused=True)
        return bq - g[0], bqd - g[1], self.scatter(lam, qd.shape[0]), -g[2]


def exact(case, seed):
    links = {"pendulum": 2, "chains": case["links"], "trees": case["links"], "humanoid": 8}.get(case["family"], 5)
    passes = 1 if case["kind"] == "step" else 3 if case["kind"] == "jvp" else 4
    if case["family"] == "quadruped_contact" or case["T"] * links * passes * (0.0012 + 4e-8 * case["B"]) > 10:
        return None
    w = _work_of(case, seed)
    dev = torch.device("cuda")
    x = {n: y.double() for n, y in _inputs(case, seed, w, dev).items()}
    m = _Plain(w.model, dev)
    q, qd, tau, mass = x["q0"], x["qd0"], x["tau"], x["mass"]
    if case["kind"] in ("step", "jvp"):
        mass = torch.as_tensor(w.model.mass, device=dev)
    if case["kind"] == "step":
        q, qd = m.step(q, qd, tau[0], mass)
        return {"q": q, "qd": qd}
    if case["kind"] == "jvp":
        (q, qd), (dq, dqd) = torch.func.jvp(lambda *y: m.step(*y, mass), (q, qd, tau[0]), (x["dq"], x["dqd"], x["dtau"]))
        return {"q": q, "qd": qd, "dq": dq, "dqd": dqd}
    states = [(q, qd)]
    for t in range(case["T"]):
        states.append(m.step(*states[-1], tau[t], mass))
    traj = torch.stack([torch.cat(s) for s in states])
    nq = q.shape[0]
    gx = x.get("gx")
    g = (gx[-1, :nq], gx[-1, nq:]) if gx is not None else (x["gq"], x["gqd"])
    gtau, gmass = torch.zeros_like(tau), torch.zeros_like(mass)
    for t in range(case["T"] - 1, -1, -1):
        bq, bqd, gtau[t], bm = m.pull_back(*states[t], tau[t], mass, *g)
        gmass += bm
        g = (bq, bqd) if gx is None else (bq + gx[t, :nq], bqd + gx[t, nq:])
    out = {"traj": traj} if gx is not None else {"qT": states[-1][0], "qdT": states[-1][1]}
    out.update(zip(("gq0", "gqd0", "gtau", "gmass"), (g[0], g[1], gtau, gmass)))
    return out
