"""What is timed: the calls that a user of this library makes, at the sizes of
its own workloads (workloads.py, the benchmark and the tests).

A case is one call, or one forward and backward, on one tree at one batch
size. Trees: the 7-DOF arm, the 11-DOF spined quadruped, legged robots of 12
and 18 DOF, the humanoid on a fixed base (23 DOF) and floating (29 DOF). Models
keep the default launch settings; "specialize" compiles the kernel kinds that
the call uses for the tree, as the README's example does for all kinds.
Inputs have the distributions of workloads.random_state: joint positions over
the whole circle, unit-variance velocities and accelerations, torques of
standard deviation 5, a free base at a random pose.

`exact` restates every result in plain torch, in 64 bits: textbook recursions
on 3-vectors, derivatives by torch.autograd, forward dynamics by a Cholesky
solve of the joint-space mass matrix.
"""
from __future__ import annotations

import functools

import numpy as np
import torch

from paper_2605_31481_gb300 import api, autograd, costs
from paper_2605_31481_gb300 import workloads as w

TREES = {
    "arm7": lambda: w.chain(7, seed=0),
    "quadruped11": lambda: w.spined_quadruped(seed=0),
    "legged12": lambda: w.legged(4, seed=0),
    "legged18": lambda: w.legged(6, seed=0),
    "humanoid23": lambda: w.humanoid(seed=0, floating=False),
    "humanoid29": lambda: w.humanoid(seed=0, floating=True),
}

# the kernel kinds that a call uses, for models that are specialised
KINDS = {"step": ("eval",), "control": ("eval",), "rl": ("eval",), "sysid": ("loss_grad",), "aba": ("aba",),
         "train_id": ("rnea", "rnea_vjp"), "train_fd": ("aba", "aba_vjp"), "linearize_fd": ("aba_derivatives",),
         "linearize_id": ("rnea_derivatives",), "ik": ("jacobian", "fk", "fk_vjp")}

# the mixed batch's share of environments per tree (of the benchmark's 4096, 2048, 1024, 512 and 256)
MIX = (16, 8, 4, 2, 1)


def listed():
    return [
        # one arm in a control loop: poses, end-effector Jacobian, inverse dynamics and mass matrix; latency only
        {"name": "control_arm7_b1", "op": "control", "tree": "arm7", "B": 1, "specialize": True},
        # the benchmark's step: all five operators on the quadruped, a common RL batch
        {"name": "step_quadruped11_b4096", "op": "step", "tree": "quadruped11", "B": 4096, "specialize": True},
        # the same on the floating humanoid, without run-time compilation, at a large RL batch
        {"name": "step_humanoid29_b16384", "op": "step", "tree": "humanoid29", "B": 16384, "specialize": False},
        # the controller step of an RL loop with the inverse dynamics' gradient in the same launch
        {"name": "rl_quadruped11_b4096", "op": "rl", "tree": "quadruped11", "B": 4096, "specialize": True},
        # one iteration of system identification: torque loss and its gradient in all 70 parameters
        {"name": "sysid_arm7_b8192", "op": "sysid", "tree": "arm7", "B": 8192, "specialize": True},
        # forward dynamics of a large simulation batch
        {"name": "aba_humanoid29_b65536", "op": "aba", "tree": "humanoid29", "B": 65536, "specialize": False},
        # inverse dynamics forward and backward through autograd, the inertias learnt too
        {"name": "train_id_humanoid29_b65536", "op": "train_id", "tree": "humanoid29", "B": 65536,
         "specialize": False},
        # differentiable simulation with a hand-written backward: forward dynamics and its adjoint, a ragged batch
        {"name": "train_fd_quadruped11_b5001", "op": "train_fd", "tree": "quadruped11", "B": 5001,
         "specialize": True},
        # linearised forward dynamics of a trajectory optimiser: knots x environments
        {"name": "linearize_fd_legged12_b1000", "op": "linearize_fd", "tree": "legged12", "B": 1000,
         "specialize": False},
        # dense derivatives of inverse dynamics of the humanoid
        {"name": "linearize_id_humanoid29_b2048", "op": "linearize_id", "tree": "humanoid29", "B": 2048,
         "specialize": False},
        # inverse kinematics by gradient: feet and hands' Jacobians, poses forward and backward
        {"name": "ik_humanoid23_b3000", "op": "ik", "tree": "humanoid23", "B": 3000, "specialize": False},
        # the benchmark's mixed batch of five robots in one launch
        {"name": "mixed_b7936", "op": "mixed", "tree": "mixed", "B": 7936, "specialize": False},
    ]


# ranges of the drawn cases: the trees of each call, its smallest batch, and the most bodies x environments
RANGES = {
    "control": (("arm7", "quadruped11", "legged12"), 1, 12 * 256, True),
    "step": (("arm7", "quadruped11", "legged18", "humanoid29"), 16, 24 * 16384, False),
    "rl": (("arm7", "quadruped11", "legged12"), 64, 11 * 16384, True),
    "sysid": (("arm7", "quadruped11", "legged12"), 256, 7 * 32768, True),
    "aba": (("arm7", "legged18", "humanoid23", "humanoid29"), 32, 24 * 65536, False),
    "train_id": (("arm7", "legged18", "humanoid29"), 64, 24 * 65536, False),
    "train_fd": (("arm7", "quadruped11", "legged12"), 64, 11 * 16384, True),
    "linearize_fd": (("arm7", "legged12", "humanoid23"), 16, 12 * 2048, False),
    "linearize_id": (("quadruped11", "legged18", "humanoid29"), 16, 24 * 2048, False),
    "ik": (("arm7", "legged18", "humanoid23"), 16, 23 * 16384, False),
    "mixed": (("mixed",), 128, 16 * 16384, False),
}


def draw(rng):
    op = rng.choice(sorted(RANGES))
    trees, lo, most, spec = RANGES[op]
    tree = rng.choice(trees)
    n = 16 if tree == "mixed" else TREES[tree]().n_bodies
    hi = most // n
    B = int(round(lo * (hi / lo) ** rng.random()))
    return {"op": op, "tree": tree, "B": max(lo, min(hi, B)), "specialize": spec and tree in ("arm7", "quadruped11")}


# ---------------------------------------------------------------------------
# what a program has in hand, and its call
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _tree(name):
    return TREES[name]()


@functools.lru_cache(maxsize=None)
def _model(name, kinds):
    """A program makes a robot's model once and keeps it."""
    return api.Model(_tree(name), specialize=list(kinds) if kinds else False)


@functools.lru_cache(maxsize=None)
def _mixed():
    trees = w.mixed_trees()
    return trees, api.MultiBatch([api.Model(t) for t in trees])


def _counts(B):
    c = [max(1, B * s // sum(MIX)) for s in MIX]
    c[0] += max(0, B - sum(c))
    return c


def _state(tree, B, gen):
    dev = "cuda"
    q = (torch.rand(tree.nq, B, generator=gen, device=dev) * 2 - 1) * np.pi
    for i, t in enumerate(tree.jtype):
        if int(t) == w.FREE:
            k = int(tree.q_index()[i])
            q[k:k + 3] = torch.randn(3, B, generator=gen, device=dev)
            quat = torch.randn(4, B, generator=gen, device=dev)
            q[k + 3:k + 7] = quat / quat.norm(dim=0)
    qd, qdd = (torch.randn(tree.nv, B, generator=gen, device=dev) for _ in range(2))
    tau = 5 * torch.randn(tree.nv, B, generator=gen, device=dev)
    return {"q": q, "qd": qd, "qdd": qdd, "tau": tau}


def _theta(tree):
    """Inertial parameters about the body origin, 64 bits: m, m c, I_com + m (|c|^2 1 - c c^T)."""
    m, c = tree.mass, tree.com
    x, y, z = c.T
    I6 = tree.I_com + m[:, None] * np.stack([y * y + z * z, -x * y, x * x + z * z, -x * z, -y * z, x * x + y * y], 1)
    return np.concatenate([m[:, None], m[:, None] * c, I6], 1)


def _inputs(case, seed):
    """The call's tensors by name, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    op, B = case["op"], int(case["B"])
    if op == "mixed":
        return {"items": [_state(t, n, gen) for t, n in zip(w.mixed_trees(), _counts(B))]}
    tree = _tree(case["tree"])
    x = _state(tree, B, gen)
    if op in ("sysid", "train_id"):
        th = torch.from_numpy(_theta(tree).astype(np.float32)).cuda()
        x["theta"] = th * (1 + 0.3 * (2 * torch.rand(th.shape, generator=gen, device="cuda") - 1))
    if op in ("train_id", "train_fd"):
        x["bar"] = torch.randn(tree.nv, B, generator=gen, device="cuda")
    if op == "ik":
        x["bar"] = torch.randn(tree.n_bodies, 12, B, generator=gen, device="cuda")
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    op, B = case["op"], int(case["B"])
    st = {"op": op, "x": x}
    if op == "mixed":
        _, st["multi"] = _mixed()
        new = lambda *shape: torch.empty(*shape, device="cuda")  # noqa: E731
        for m, s in zip(st["multi"].models, x["items"]):
            B = s["q"].shape[1]
            out = {"poses": new(m.n_bodies, 12, B), "tau": new(m.nv, B), "M": new(m.nv, m.nv, B), "qdd": new(m.nv, B)}
            st.setdefault("items", []).append({**s, "fk": True, "rnea": True, "crba": True, "aba": True, "out": out})
        return st
    tree = _tree(case["tree"])
    st["model"] = m = _model(case["tree"], KINDS[op] if case.get("specialize") else None)
    st["links"] = list(tree.ee)
    new = lambda *shape: torch.empty(*shape, device="cuda")  # noqa: E731
    if op in ("step", "control", "rl"):  # a control loop keeps its output buffers
        st["out"] = {"poses": new(m.n_bodies, 12, B), "J": new(len(tree.ee), 6, m.nv, B), "tau": new(m.nv, B)}
        if op != "rl":
            st["out"]["M"] = new(m.nv, m.nv, B)
        if op == "step":
            st["out"]["qdd"] = new(m.nv, B)
        if op == "rl":
            st["out"].update(q_bar=new(m.nq, B), qd_bar=new(m.nv, B))
    if op == "sysid":
        st["scratch"] = api.adjoint_scratch(m, B)
        st["buf"] = new(m.n_bodies * 10 + 1)
    if op == "train_id":
        for k in ("q", "qd", "qdd", "theta"):
            x[k].requires_grad_()
    return st


def run(state):
    op, x, m = state["op"], state["x"], state.get("model")
    if op == "mixed":
        return state["multi"].eval(state["items"])
    if op == "control":
        return api.eval(m, x["q"], x["qd"], x["qdd"], fk=True, links=state["links"], rnea=True, crba=True,
                        out=state["out"])
    if op == "step":
        return api.eval(m, x["q"], x["qd"], x["qdd"], x["tau"], fk=True, links=state["links"], rnea=True, crba=True,
                        aba=True, out=state["out"])
    if op == "rl":
        return api.eval(m, x["q"], x["qd"], x["qdd"], fk=True, links=state["links"], rnea=True, q_bar=True,
                        qd_bar=True, tau_bar="tau", out=state["out"])
    if op == "sysid":
        loss, grad, _, _ = api.rnea_loss_grad(m, x["q"], x["qd"], x["qdd"], x["tau"], theta=x["theta"],
                                              scratch=state["scratch"], out=state["buf"])
        return {"loss": loss, "theta": grad}
    if op == "aba":
        return {"qdd": api.aba(m, x["q"], x["qd"], x["tau"])}
    if op == "train_id":
        tau = autograd.rnea(m, x["q"], x["qd"], x["qdd"], x["theta"])
        g = torch.autograd.grad(tau, (x["q"], x["qd"], x["qdd"], x["theta"]), x["bar"])
        return {"tau": tau, "q": g[0], "qd": g[1], "qdd": g[2], "theta": g[3]}
    if op == "train_fd":
        qdd = api.aba(m, x["q"], x["qd"], x["tau"])
        g = api.aba_vjp(m, x["q"], x["qd"], qdd, x["bar"], theta_bar=False)
        return {"qdd": qdd, "q": g["q"], "qd": g["qd"], "tau": g["tau"]}
    if op == "linearize_fd":
        return api.aba_derivatives(m, x["q"], x["qd"], x["tau"], qdd=True)
    if op == "linearize_id":
        return api.rnea_derivatives(m, x["q"], x["qd"], x["qdd"])
    if op == "ik":
        return {"J": api.jacobian(m, x["q"], state["links"]), "poses": api.fk(m, x["q"]),
                "q": api.fk_vjp(m, x["q"], x["bar"])}
    raise ValueError(op)


# ---------------------------------------------------------------------------
# what the path cannot do without
# ---------------------------------------------------------------------------

def _work(tree, op, B):
    """(bytes, flops) of one environment. Adjoints: twice the forward arithmetic beside the forward sweep.
    Derivatives: per direction, a tangent through the subtree below it and up the path above it."""
    nq, nv, nb = tree.nq, tree.nv, tree.n_bodies
    ee = list(tree.ee)
    fl = lambda *ops: sum(costs.flops(tree, o, ee) for o in ops)  # noqa: E731
    J = 6 * nv * len(ee)
    path = [len(costs._path(tree, i)) for i in range(nb)]
    dofs = nv * (sum(path) / nb)  # direction-body pairs along support paths, upwards and downwards alike
    if op == "control":
        return nq + 2 * nv + 12 * nb + J + nv + nv * nv, fl("jacobian", "rnea", "crba")
    if op == "step":
        return nq + 3 * nv + 12 * nb + J + nv + nv * nv + nv, fl("jacobian", "rnea", "crba", "aba")
    if op == "rl":
        return nq + 2 * nv + 12 * nb + J + nv + nq + nv, fl("jacobian") + 3 * fl("rnea")
    if op == "sysid":
        return nq + 3 * nv, 3 * fl("rnea")
    if op == "aba":
        return nq + 3 * nv, fl("aba")
    if op == "train_id":  # forward, then backward: each reads its inputs
        return (nq + 3 * nv) + (nq + 3 * nv) + (nq + 2 * nv), 4 * fl("rnea")
    if op == "train_fd":
        return (nq + 3 * nv) + (nq + 3 * nv) + (nq + 2 * nv), 2 * fl("aba") + 3 * fl("rnea")
    if op == "linearize_id":
        return nq + 2 * nv + 2 * nv * nv, fl("rnea") + dofs * 2 * 300
    if op == "linearize_fd":
        return nq + 3 * nv + 3 * nv * nv, fl("aba", "rnea", "crba") + dofs * 2 * 300 + nv ** 3 * 5
    if op == "ik":
        return nq + J + nq + 12 * nb + nq + 12 * nb + nq, fl("jacobian") + 3 * fl("fk")
    raise ValueError(op)


def work(case):
    B = int(case["B"])
    if case["op"] == "mixed":
        by, fl = 0.0, 0.0
        for t, n in zip(w.mixed_trees(), _counts(B)):
            by += 4.0 * n * (t.nq + 3 * t.nv + 12 * t.n_bodies + t.nv + t.nv * t.nv + t.nv)
            fl += n * sum(costs.flops(t, o) for o in ("fk", "rnea", "crba", "aba"))
        return {"bytes": by, "flops": float(fl)}
    floats, flops = _work(_tree(case["tree"]), case["op"], B)
    return {"bytes": 4.0 * floats * B, "flops": float(flops) * B}


# ---------------------------------------------------------------------------
# the results in 64 bits
# ---------------------------------------------------------------------------

def _skew(v):
    x, y, z = v.unbind(-1)
    o = torch.zeros_like(x)
    return torch.stack([o, -z, y, z, o, -x, -y, x, o], -1).view(*v.shape[:-1], 3, 3)


def _mv(R, v):
    return (R @ v.unsqueeze(-1)).squeeze(-1)


def _tv(R, v):
    return (R.transpose(-1, -2) @ v.unsqueeze(-1)).squeeze(-1)


def _x(a, b):
    a, b = torch.broadcast_tensors(a, b)
    return torch.linalg.cross(a, b)


class _Exact:
    """One tree's recursions on (..., features) tensors of 64 bits (T_link is the identity in every tree here)."""

    def __init__(self, tree):
        c = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float64)).cuda()  # noqa: E731
        self.t, self.axis, self.Tj = tree, c(tree.axis), c(tree.T_joint)
        self.qi, self.vi = tree.q_index(), tree.v_index()
        self.theta = c(_theta(tree))
        self.g = c(tree.gravity)

    def joints(self, q, d=None):
        """(R, t) of each body in its parent, at q moved along the tangent d."""
        out = []
        eye = torch.eye(3, dtype=torch.float64, device=q.device)
        for i, ty in enumerate(self.t.jtype):
            R0, t0 = self.Tj[i, :9].view(3, 3), self.Tj[i, 9:]
            k, v = int(self.qi[i]), int(self.vi[i])
            if int(ty) == w.FREE:
                p, quat = q[..., k:k + 3], q[..., k + 3:k + 7]
                quat = quat / quat.norm(dim=-1, keepdim=True)
                K = _skew(quat[..., :3])
                R = eye + 2 * quat[..., 3, None, None] * K + 2 * K @ K
                if d is not None:
                    p = p + _mv(R, d[..., v:v + 3])
                    R = R @ (eye + _skew(d[..., v + 3:v + 6]))
                out.append((R0 @ R, _mv(R0, p) + t0))
            else:
                a = q[..., k] if d is None else q[..., k] + d[..., v]
                K = _skew(self.axis[i])
                R = eye + torch.sin(a)[..., None, None] * K + (1 - torch.cos(a))[..., None, None] * (K @ K)
                out.append((R0 @ R, t0.expand(*a.shape, 3)))
        return out

    def poses(self, q):
        W = []
        for i, (R, t) in enumerate(self.joints(q)):
            p = int(self.t.parent[i])
            W.append((R, t) if p < 0 else (W[p][0] @ R, _mv(W[p][0], t) + W[p][1]))
        return W

    def motion(self, i, x):
        """S_i x as (w, v); the free joint's coordinates are [v; w]."""
        v = int(self.vi[i])
        if int(self.t.jtype[i]) == w.FREE:
            return x[..., v + 3:v + 6], x[..., v:v + 3]
        a = x[..., v, None] * self.axis[i]
        return a, torch.zeros_like(a)

    def rnea(self, X, qd, qdd, theta=None, gravity=True):
        th = self.theta if theta is None else theta
        n = self.t.n_bodies
        V, A, F = [], [], []
        for i in range(n):
            R, t = X[i]
            p = int(self.t.parent[i])
            sw, sv = self.motion(i, qd)
            aw, av = self.motion(i, qdd)
            if p < 0:
                g = _tv(R, -self.g if gravity else torch.zeros_like(self.g))
                wi, vi, dw, dv = sw, sv, aw, av + g
            else:
                (pw, pv), (qw, qv) = V[p], A[p]
                wi, vi = _tv(R, pw) + sw, _tv(R, pv - _x(t, pw)) + sv
                dw = _tv(R, qw) + aw + _x(wi, sw)
                dv = _tv(R, qv - _x(t, qw)) + av + _x(wi, sv) + _x(vi, sw)
            I, h, mass = th[i, 4:], th[i, 1:4], th[i, 0]
            Io = torch.stack([I[0], I[1], I[3], I[1], I[2], I[4], I[3], I[4], I[5]]).view(3, 3)
            hw, hv = _mv(Io, wi) + _x(h, vi), mass * vi - _x(h, wi)
            fw = _mv(Io, dw) + _x(h, dv) + _x(wi, hw) + _x(vi, hv)
            fv = mass * dv - _x(h, dw) + _x(wi, hv)
            V.append((wi, vi)), A.append((dw, dv)), F.append((fw, fv))
        tau = [None] * n
        for i in range(n - 1, -1, -1):
            fw, fv = F[i]
            tau[i] = torch.cat([fv, fw], -1) if int(self.t.jtype[i]) == w.FREE else (fw * self.axis[i]).sum(-1, True)
            p = int(self.t.parent[i])
            if p >= 0:
                R, t = X[i]
                lv = _mv(R, fv)
                F[p] = (F[p][0] + _mv(R, fw) + _x(t, lv), F[p][1] + lv)
        return torch.cat(tau, -1)

    def mass_matrix(self, X, B):
        """(B, nv, nv): column k is inverse dynamics at a unit acceleration without gravity."""
        nv = self.t.nv
        e = torch.eye(nv, dtype=torch.float64, device="cuda")[:, None, :].expand(nv, B, nv)
        return self.rnea(X, torch.zeros_like(e), e, gravity=False).permute(1, 2, 0)

    def aba(self, q, qd, tau):
        """(qdd, Cholesky factor of M)."""
        X = self.joints(q)
        L = torch.linalg.cholesky(self.mass_matrix(X, q.shape[0]))
        bias = self.rnea(X, qd, torch.zeros_like(qd))
        return torch.cholesky_solve((tau - bias).unsqueeze(-1), L).squeeze(-1), L

    def jacobian(self, q, links):
        """(n_links, 6, nv, B): world twists [v; w] at the world origin."""
        W = self.poses(q)
        J = torch.zeros(len(links), 6, self.t.nv, q.shape[0], dtype=torch.float64, device="cuda")
        for l, b in enumerate(links):
            for k in costs._path(self.t, b):
                R, p = W[k]
                v = int(self.vi[k])
                if int(self.t.jtype[k]) == w.FREE:
                    for j in range(3):
                        J[l, :3, v + j] = R[..., j].T
                        J[l, 3:, v + 3 + j] = R[..., j].T
                        J[l, :3, v + 3 + j] = _x(p, R[..., j]).T
                else:
                    a = _mv(R, self.axis[k])
                    J[l, 3:, v], J[l, :3, v] = a.T, _x(p, a).T
        return J

    def fk(self, q):
        return torch.stack([torch.cat([R.reshape(*R.shape[:-2], 9), t], -1) for R, t in self.poses(q)], -2)

    def derivatives(self, q, qd, qdd):
        """d tau / d q (tangent) and d tau / d qd, (B, nv, nv) each."""
        d = torch.zeros_like(qd, requires_grad=True)
        qd = qd.detach().requires_grad_()
        tau = self.rnea(self.joints(q, d), qd, qdd)
        rows = [torch.autograd.grad(tau[:, r].sum(), (d, qd), retain_graph=True) for r in range(self.t.nv)]
        return torch.stack([r[0] for r in rows], 1), torch.stack([r[1] for r in rows], 1)


def _soa(x):
    return x.movedim(0, -1).contiguous()


def _forward(E, s, links, ops):
    """The five operators' results for one chunk of environments (feature-last inputs)."""
    q, qd, qdd, tau = s
    out = {}
    X = E.joints(q)
    if "poses" in ops:
        out["poses"] = _soa(E.fk(q))
    if "J" in ops:
        out["J"] = E.jacobian(q, links)
    if "tau" in ops:
        out["tau"] = _soa(E.rnea(X, qd, qdd))
    if "M" in ops:
        out["M"] = _soa(E.mass_matrix(X, q.shape[0]))
    if "qdd" in ops:
        out["qdd"] = _soa(E.aba(q, qd, tau)[0])
    return out


def _chunks(x, size=8192):
    x = {k: v.double() for k, v in x.items() if k in ("q", "qd", "qdd", "tau")}
    for lo in range(0, x["q"].shape[1], size):
        yield [x[k][:, lo:lo + size].T for k in ("q", "qd", "qdd", "tau")], slice(lo, lo + size)


def _joined(parts):
    return {k: torch.cat([p[k] for p in parts], -1) for k in parts[0]}


def exact(case, seed):
    x = _inputs(case, seed)
    op = case["op"]
    if op == "mixed":
        ops = ("poses", "tau", "M", "qdd")
        return [_joined([_forward(_Exact(t), s, (), ops) for s, _ in _chunks(item)])
                for t, item in zip(w.mixed_trees(), x["items"])]
    tree = _tree(case["tree"])
    E, links = _Exact(tree), list(tree.ee)
    if op in ("control", "step"):
        ops = ("poses", "J", "tau", "M") + (("qdd",) if op == "step" else ())
        return _joined([_forward(E, s, links, ops) for s, _ in _chunks(x)])
    if op == "aba":
        return _joined([_forward(E, s, links, ("qdd",)) for s, _ in _chunks(x)])
    if op == "linearize_id":
        parts = []
        for (q, qd, qdd, _), _ in _chunks(x):
            dq, dqd = E.derivatives(q, qd, qdd)
            parts.append({"q": _soa(dq), "qd": _soa(dqd)})
        return _joined(parts)
    if op == "linearize_fd":
        parts = []
        for (q, qd, _, tau), _ in _chunks(x):
            qdd, L = E.aba(q, qd, tau)
            dq, dqd = E.derivatives(q, qd, qdd)
            eye = torch.eye(tree.nv, dtype=torch.float64, device="cuda").expand_as(L)
            parts.append({"tau": _soa(torch.cholesky_solve(eye, L)), "q": _soa(-torch.cholesky_solve(dq, L)),
                          "qd": _soa(-torch.cholesky_solve(dqd, L)), "qdd": _soa(qdd)})
        return _joined(parts)
    if op == "ik":
        parts = []
        for (q, _, _, _), part in _chunks(x):
            q = q.detach().requires_grad_()
            P = E.fk(q)
            (g,) = torch.autograd.grad(P, (q,), x["bar"][..., part].double().movedim(-1, 0))
            parts.append({"J": E.jacobian(q.detach(), links), "poses": _soa(P.detach()), "q": _soa(g)})
        return _joined(parts)
    # the adjoints of inverse dynamics: a sum over environments in the parameters
    th = (x["theta"].double() if "theta" in x else E.theta).detach().requires_grad_()
    parts, loss, gth = [], 0.0, torch.zeros_like(th)
    for (q, qd, qdd, tau), part in _chunks(x):
        L = None
        if op == "train_fd":
            with torch.no_grad():
                qdd, L = E.aba(q, qd, tau)
        q, qd, qdd = (t.detach().requires_grad_() for t in (q, qd, qdd))
        r = E.rnea(E.joints(q), qd, qdd, th)
        if op == "sysid":
            f = (r - tau).square().sum()
            loss = loss + f.detach()
            gth += torch.autograd.grad(f, (th,))[0]
            continue
        if op == "rl":  # the cotangent is the torque itself
            g = torch.autograd.grad(r, (q, qd), r.detach())
            parts.append({"poses": _soa(E.fk(q.detach())), "J": E.jacobian(q.detach(), links),
                          "tau": _soa(r.detach()), "q_bar": _soa(g[0]), "qd_bar": _soa(g[1])})
            continue
        bar = x["bar"][:, part].double().T
        if op == "train_fd":
            lam = torch.cholesky_solve(bar.unsqueeze(-1), L).squeeze(-1)
            g = torch.autograd.grad(r, (q, qd), -lam)
            parts.append({"qdd": _soa(qdd.detach()), "q": _soa(g[0]), "qd": _soa(g[1]), "tau": _soa(lam)})
        else:
            g = torch.autograd.grad(r, (q, qd, qdd, th), bar)
            gth += g[3]
            parts.append({"tau": _soa(r.detach()), "q": _soa(g[0]), "qd": _soa(g[1]), "qdd": _soa(g[2])})
    if op == "sysid":
        return {"loss": loss, "theta": gth}
    out = _joined(parts)
    if op == "train_id":
        out["theta"] = gth
    return out
