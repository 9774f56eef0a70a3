"""What a user of this framework has it compute, as cases to be timed: single
steps, autograd steps, open-loop windows (forward and adjoint), episodic
windows, policy windows and critic targets, on the models and at the sizes of
the workloads in ``inputs`` and of the bench's window-length study.

A window gradient in ground contact jumps by a finite amount where a contact,
friction or joint-limit switch is decided by rounding (the derivatives of those
forces are discontinuous).  With seeded initial states, all feet 2 mm in the
ground, no switch is near for the first steps; later ones are.  So the cases
that return gradients in contact take short windows, and the longer windows are
free of contact: the cart-pole at h = 32, and the ant-like model dropped from
2 m (the same kernels and contact tests, no touch-down within the window) at the
study's h = 8, past which its random torques amplify a last-bit difference to
more than 1e-5 of the gradient.  The muscle, humanoid and half-cheetah models'
windows with gradients are dropped too: their first steps already meet switches.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2204_07137_gb300 import inputs
from paper_2204_07137_gb300.policy import PolicyMLP, observation_size, policy_window_loss
from paper_2204_07137_gb300.shac import td_lambda
from paper_2204_07137_gb300.sim import SimStep, SimWindow, Simulator

GAMMA, LAMBDA = 0.99, 0.95


def listed():
    return [
        # One control step of the smallest model at the paper's N = 64: a rollout or evaluation loop, launch-bound.
        dict(name="step cartpole 64", kind="step", groups="cartpole:64", h=1, drop=0.0, special=False),
        # One step and its backward through the autograd layer, N = 64: what the learner does 32 times an episode.
        dict(name="autograd step ant 64", kind="autograd", groups="ant:64", h=1, drop=0.0, special=False),
        # Critic targets of a full batch's window (Eq. td-lambda).
        dict(name="td-lambda 32x2048", kind="td", h=32, n=2048, done=True),
        # A whole training window of the smallest workload, captured in a CUDA graph as the bench does.
        dict(name="graph window cartpole 64 h32", kind="graph", groups="cartpole:64", h=32, drop=0.0, special=True),
        # The headline batch: 2048 ant-like environments, kernels specialised for the model.
        dict(name="window ant 2048 h8", kind="window", groups="ant:2048", h=8, drop=2.0, special=True, tape=False),
        # A ragged batch on the ground with the generic kernels (what a program runs that compiles nothing).
        dict(name="window ant 1531 h2", kind="window", groups="ant:1531", h=2, drop=0.0, special=False, tape=False),
        # The window-length study's many-environment end, substep records kept in memory: throughput.
        dict(name="tape window ant 16384 h4", kind="window", groups="ant:16384", h=4, drop=2.0, special=True, tape=True),
        # Evaluation rollout of the humanoid-like workload: forward only, in contact.
        dict(name="rollout humanoid 1024 h8", kind="rollout", groups="humanoid:1024", h=8, drop=0.0, special=False),
        # The heterogeneous workload: three models in one launch per direction.
        dict(name="window hetero h2", kind="window", groups="cartpole:4096,ant:2048,humanoid:1024", h=2, drop=1.0, special=False, tape=False),
        # The muscle-actuated workload (152 muscles), open loop.
        dict(name="window mtu 512 h2", kind="window", groups="mtu:512", h=2, drop=1.0, special=True, tape=False),
        # Early termination and resets inside the window, gradient cut at them; an odd batch of a planar model.
        dict(name="episodic hopper 777 h4", kind="episodic", groups="hopper:777", h=4, drop=0.0, special=False),
        # The muscle workload with its policy in the loop: loss and parameter gradients.
        dict(name="policy mtu 512 h2", kind="policy", groups="mtu:512", h=2, drop=0.0, special=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _clear(model):
    """Drop height of a model whose gradients in contact are undecided from the first steps on."""
    return 1.0 if model in ("humanoid", "mtu", "halfcheetah") else 0.0


def draw(rng):
    kind = rng.choice(["step", "autograd", "td", "graph", "window", "flight", "rollout", "hetero", "episodic", "policy"])
    special = rng.random() < 0.5
    if kind == "td":
        return dict(kind="td", h=_log_int(rng, 4, 128), n=_log_int(rng, 64, 65536), done=rng.random() < 0.5)
    if kind == "step":
        return dict(kind="step", groups="%s:%d" % (rng.choice(["cartpole", "ant", "halfcheetah", "hopper", "humanoid"]), _log_int(rng, 1, 1024)), h=1,
                    drop=0.0, special=special)
    if kind == "autograd":
        model, most = rng.choice([("cartpole", 1024), ("ant", 1024), ("halfcheetah", 1024), ("hopper", 1024), ("humanoid", 64)])
        return dict(kind="autograd", groups="%s:%d" % (model, _log_int(rng, 4, most)), h=1, drop=_clear(model), special=special)
    if kind == "graph":
        return dict(kind="graph", groups="cartpole:%d" % _log_int(rng, 16, 4096), h=_log_int(rng, 4, 32), drop=0.0, special=special)
    if kind == "flight":
        n = _log_int(rng, 64, 8192)
        return dict(kind="window", groups="ant:%d" % n, h=min(_log_int(rng, 2, 8), 32768 // n), drop=2.0, special=special, tape=rng.random() < 0.5)
    if kind == "window":
        model, n, h = rng.choice([("ant", 2048, 2), ("halfcheetah", 2048, 2), ("hopper", 1024, 2), ("mtu", 256, 2)])
        return dict(kind="window", groups="%s:%d" % (model, _log_int(rng, 16, n)), h=rng.randint(1, h), drop=_clear(model), special=special,
                    tape=rng.random() < 0.3)
    if kind == "rollout":
        model, n = rng.choice([("humanoid", 512), ("ant", 4096), ("halfcheetah", 4096), ("hopper", 4096), ("mtu", 128)])
        return dict(kind="rollout", groups="%s:%d" % (model, _log_int(rng, 32, n)), h=rng.randint(2, 8), drop=0.0, special=special)
    if kind == "hetero":
        return dict(kind="window", groups="cartpole:%d,ant:%d,humanoid:%d" % (_log_int(rng, 16, 4096), _log_int(rng, 16, 2048), _log_int(rng, 16, 1024)),
                    h=rng.randint(1, 2), drop=1.0, special=False, tape=rng.random() < 0.3)
    if kind == "episodic":
        return dict(kind="episodic", groups="hopper:%d" % _log_int(rng, 32, 777), h=rng.randint(2, 4), drop=0.0, special=special)
    return dict(kind="policy", groups="mtu:%d" % _log_int(rng, 16, 512), h=rng.randint(1, 2), drop=0.0, special=special)


def _groups(case):
    return [(getattr(inputs, name)(), int(n)) for name, n in (g.split(":") for g in case["groups"].split(","))]


def _arrays(case, seed):
    """Per group: q0 [nq, N], qd0 [nv, N], act [h, na, N] and the cotangents of
    the final state; the reward cotangents [h, n_envs] of the discounted mean."""
    groups, out = _groups(case), []
    total, h = sum(n for _, n in groups), case["h"]
    for k, (m, n) in enumerate(groups):
        rng = np.random.default_rng([seed, k])
        q, qd = inputs.initial_state(m, n, seed)
        if case["drop"]:
            qd += rng.uniform(-0.5, 0.5, qd.shape).astype(np.float32)     # mid-motion
            if int(m.joint_type[0]) == inputs.FREE:
                q[2] += np.float32(case["drop"])
            elif m.height_q >= 0:
                q[m.height_q] += np.float32(case["drop"])
        bar = [(0.1 / (total * h) * rng.standard_normal(x.shape)).astype(np.float32) for x in (q, qd)]   # of the terminal value
        out.append((q, qd, inputs.window_actions(m, n, h, seed), *bar))
    rb = np.repeat(-(GAMMA ** np.arange(h, dtype=np.float64))[:, None] / (total * h), total, 1).astype(np.float32)
    return groups, out, rb


def _flat(parts, lead=()):
    return torch.from_numpy(np.concatenate([np.ascontiguousarray(p).reshape(*lead, -1) for p in parts], -1)).cuda()


def _td_arrays(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    h, n = case["h"], case["n"]
    r, v = torch.randn(h, n, device="cuda", generator=g), torch.randn(h + 1, n, device="cuda", generator=g)
    d = (torch.rand(h, n, device="cuda", generator=g) < 0.05).to(torch.uint8) if case["done"] else None
    return r, v, d


def _reset_arrays(case, seed, m, n):
    qr, qdr = inputs.initial_state(m, n, seed + 1)
    return qr, qdr, np.random.default_rng([seed, 99]).integers(0, 6, n).astype(np.int32)


HORIZON = 6      # episode length of the episodic cases: a third of the environments or more end within the window


def _policy(case, m, seed):
    g = torch.Generator().manual_seed(seed)
    return PolicyMLP(observation_size(m), m.na, generator=g, muscles=m.n_muscles > 0).cuda()


def prepare(case, seed):
    if case["kind"] == "td":
        return dict(kind="td", args=_td_arrays(case, seed))
    groups, arrays, rb = _arrays(case, seed)
    h, kind = case["h"], case["kind"]
    sim = Simulator(groups, form="batched", h_max=h)
    if case.get("tape"):
        sim.set_window_tape(True)
    if case["special"]:
        sim.specialize()
    q, qd = (_flat([a[k] for a in arrays]) for k in (0, 1))
    act = _flat([a[2] for a in arrays], (h,))
    gq, gqd = (torch.zeros(h + 1, n, device="cuda") for n in (sim.q_size, sim.qd_size))
    gq[h], gqd[h] = (_flat([a[k] for a in arrays]) for k in (3, 4))
    s = dict(kind=kind, sim=sim, q=q, qd=qd, act=act, gq=gq, gqd=gqd, rb=torch.from_numpy(rb).cuda())
    if kind in ("autograd", "window"):
        for x in (q, qd, act):
            x.requires_grad_(True)
    if kind == "policy":
        s["net"], s["h"] = _policy(case, groups[0][0], seed), h
    if kind == "episodic":
        qr, qdr, ep = _reset_arrays(case, seed, *groups[0])
        s.update(qr=_flat([qr]), qdr=_flat([qdr]), ep=torch.from_numpy(ep).cuda(), rule=inputs.episode_rule(groups[0][0])[0])
    if kind == "graph":
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            f = sim.window_forward(q, qd, act)
            a = sim.window_adjoint(f[0], f[1], act, s["rb"], gq, gqd)
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                sim.window_forward(q, qd, act, out=f)
                sim.window_adjoint(f[0], f[1], act, s["rb"], gq, gqd, out=a)
        torch.cuda.current_stream().wait_stream(stream)
        s.update(graph=graph, out=(*f, *a))
    return s


def run(s):
    kind = s["kind"]
    if kind == "td":
        return td_lambda(*s["args"], GAMMA, LAMBDA)
    sim = s["sim"]
    if kind == "graph":
        s["graph"].replay()
        return s["out"]
    if kind == "step":
        return sim.step(s["q"], s["qd"], s["act"][0])
    if kind == "rollout":
        return sim.window_forward(s["q"], s["qd"], s["act"])
    if kind == "autograd":
        out = SimStep.apply(sim, s["q"], s["qd"], s["act"][0])
        grads = torch.autograd.grad(out, (s["q"], s["qd"], s["act"]), (s["gq"][1], s["gqd"][1], s["rb"][0]))
        return [x.detach() for x in out] + list(grads)
    if kind == "window":
        out = SimWindow.apply(sim, s["q"], s["qd"], s["act"])
        grads = torch.autograd.grad(out, (s["q"], s["qd"], s["act"]), (s["gq"], s["gqd"], s["rb"]))
        return [x.detach() for x in out] + list(grads)
    if kind == "episodic":
        ep = s["ep"].clone()
        f = sim.window_forward_episodic(s["q"], s["qd"], s["act"], s["qr"], s["qdr"], [s["rule"]], [HORIZON], ep)
        g = sim.window_adjoint_episodic(f[0], f[1], s["act"], f[3], s["rb"], s["gq"], s["gqd"])
        return [*f, *g, ep]
    loss = policy_window_loss(sim, s["net"], s["q"], s["qd"], s["h"])
    return [loss.detach(), *torch.autograd.grad(loss, list(s["net"].parameters()))]


def work(case):
    """Each input read once, each output written once; operations per substep
    of one environment from the counts of the stages (links, dense part,
    contacts, muscle segments), as the one-thread form executes them: 8.4 k
    forward and 10.8 k reverse for the ant-like model.  A gradient needs one
    forward and one reverse."""
    h = case["h"]
    if case["kind"] == "td":
        n = case["n"]
        return {"bytes": float(4 * (3 * h + 1) * n + (h * n if case["done"] else 0)), "flops": 6.0 * h * n}
    nbytes = flops = 0.0
    back = case["kind"] not in ("step", "rollout")
    for m, n in _groups(case):
        L, nv, segs = m.n_links, m.nv, len(m.via_link) - m.n_muscles
        fwd = 600 * L + nv ** 3 / 3 + 10 * nv ** 2 + 40 * m.n_contacts + 120 * segs
        rev = 1000 * L + 6 * nv ** 2 + 100 * m.n_contacts + 250 * segs
        flops += n * h * m.substeps * (fwd + (rev if back else 0))
        state, act = m.nq + m.nv, h * m.na
        nbytes += 4 * n * (state + act + (h + (case["kind"] != "step")) * state + h)
        if back:
            nbytes += 4 * n * ((h + 1) * state + h + state + act)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- 64 bits --


def _rot(x, y, z, w):
    """Rotation matrices [..., 3, 3] of unit quaternions."""
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1).unflatten(-1, (3, 3))


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _mv(A, x):
    return (A @ x.unsqueeze(-1)).squeeze(-1)


class Sim64:
    """The simulated step in 64 bits: links by composed transforms, the mass
    matrix from the Jacobians of the centres of mass, forces by the vector
    Newton-Euler recursion; derivatives by autograd."""

    def __init__(self, m, device):
        t = lambda x: torch.tensor(np.asarray(x, np.float64), device=device)  # noqa: E731
        self.m, self.L, self.nv = m, m.n_links, m.nv
        self.jt = [int(j) for j in m.joint_type]
        self.par = [int(p) for p in m.parent]
        self.qs, self.ds = m.q_start(), m.dof_start()
        quat = m.joint_quat.astype(np.float64)
        quat /= np.linalg.norm(quat, axis=1, keepdims=True)
        self.jrot = _rot(*t(quat).unbind(-1))
        axis = m.joint_axis.astype(np.float64)
        axis /= np.maximum(np.linalg.norm(axis, axis=1, keepdims=True), 1e-300)
        self.axis, self.jpos, self.com, self.mass = t(axis), t(m.joint_pos), t(m.com), t(m.mass)
        K = torch.zeros(self.L, 3, 3, dtype=torch.float64, device=device)
        for (i, j), s, k in (((0, 1), -1, 2), ((0, 2), 1, 1), ((1, 0), 1, 2), ((1, 2), -1, 0), ((2, 0), -1, 1), ((2, 1), 1, 0)):
            K[:, i, j] = s * self.axis[:, k]
        self.K, self.K2 = K, K @ K     # rotation by angle t about the axis: 1 + sin t K + (1 - cos t) K^2
        self.eye = torch.eye(3, dtype=torch.float64, device=device)
        self.inertia = t(m.inertia)[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].unflatten(-1, (3, 3))
        dof_link = [i for i, j in enumerate(self.jt) for _ in range({0: 6, 3: 0}.get(j, 1))]
        up = np.zeros((self.L, self.nv))
        for i in range(self.L):
            j = i
            while j >= 0:
                up[i, [d for d, k in enumerate(dof_link) if k == j]] = 1
                j = self.par[j]
        self.moves = t(up)                                        # [L, nv]: DOF d moves link i
        self.dof_link = torch.tensor(dof_link, device=device)
        self.spin = t([1.0 if (self.jt[k] == 1 or (self.jt[k] == 0 and d < 3)) else 0.0 for d, k in enumerate(dof_link)])
        self.arm, self.damp, self.lo, self.hi = t(m.armature), t(m.damping), t(m.q_lower), t(m.q_upper)
        self.limited = [(d, int(self.qs[k])) for d, k in enumerate(dof_link) if self.jt[k] in (1, 2)]
        self.gear = torch.zeros(m.n_tact, self.nv, dtype=torch.float64, device=device)
        for k in range(m.n_tact):
            self.gear[k, int(m.act_dof[k])] = float(m.act_gear[k])
        self.grav = t(m.gravity)
        self.c_link, self.c_pos, self.c_rad = torch.tensor(m.contact_link.astype(np.int64), device=device), t(m.contact_pos), t(m.contact_radius)
        s0 = [v for k in range(m.n_muscles) for v in range(int(m.muscle_ptr[k]), int(m.muscle_ptr[k + 1]) - 1)]
        self.seg = torch.tensor(s0, dtype=torch.int64, device=device)
        self.seg_mus = torch.tensor([k for k in range(m.n_muscles) for _ in range(int(m.muscle_ptr[k + 1]) - int(m.muscle_ptr[k]) - 1)],
                                    dtype=torch.int64, device=device)
        self.v_link, self.v_pos, self.fmax = torch.tensor(m.via_link.astype(np.int64), device=device), t(m.via_pos), t(m.muscle_fmax)
        self.h = float(np.float32(m.dt / m.substeps))
        self.rwq, self.rwqd, self.rc = t(m.rw_q), t(m.rw_qd), [float(c) for c in m.reward_coef]

    def accel(self, q, qd, a):
        N = q.shape[0]
        z = q.new_zeros(N, 3)
        R, P, W, V, AW, AV, ax, org = [], [], [], [], [], [], [], []
        for i, j in enumerate(self.jt):
            s, d, p = int(self.qs[i]), int(self.ds[i]), self.par[i]
            if j == 0:
                R.append(_rot(*q[:, s + 3:s + 7].unbind(-1)))
                P.append(q[:, s:s + 3])
                W.append(_mv(R[i], qd[:, d:d + 3]))
                V.append(_mv(R[i], qd[:, d + 3:d + 6]))
                AW.append(z)
                AV.append(_cross(W[i], V[i]))
                ax += [R[i][:, :, k] for k in range(3)] * 2
                org += [P[i]] * 6
                continue
            Rp, Pp, Wp, Vp, AWp, AVp = (R[p], P[p], W[p], V[p], AW[p], AV[p]) if p >= 0 else (self.eye.expand(N, 3, 3), z, z, z, z, z)
            Rj, r = Rp @ self.jrot[i], _mv(Rp, self.jpos[i].expand(N, 3))
            axis = _mv(Rj, self.axis[i].expand(N, 3))
            if j == 1:
                th = q[:, s, None, None]
                Rj = Rj @ (self.eye + torch.sin(th) * self.K[i] + (1 - torch.cos(th)) * self.K2[i])
            if j == 2:
                r = r + q[:, s:s + 1] * axis
            u = qd[:, d:d + 1] * axis if j in (1, 2) else z
            wr = _cross(Wp, r)
            R.append(Rj)
            P.append(Pp + r)
            W.append(Wp + u if j == 1 else Wp)
            V.append(Vp + wr + u if j == 2 else Vp + wr)
            AW.append(AWp + _cross(Wp, u) if j == 1 else AWp)
            acc = AVp + _cross(AWp, r) + _cross(Wp, wr)
            AV.append(acc + 2 * _cross(Wp, u) if j == 2 else acc)
            if j in (1, 2):
                ax.append(axis)
                org.append(P[i])
        R, P, W, V, AW, AV = (torch.stack(x, 1) for x in (R, P, W, V, AW, AV))
        ax, org = torch.stack(ax, 1), torch.stack(org, 1)
        rc = _mv(R, self.com.expand(N, -1, -1))
        C, Ac = P + rc, AV + _cross(AW, rc) + _cross(W, _cross(W, rc))
        Iw = R @ self.inertia @ R.transpose(-1, -2)
        # wrench on each link (about its centre of mass): contacts, muscles
        fn, ff = torch.zeros_like(C), torch.zeros_like(C)
        if len(self.m.contact_link):
            k = self.c_link
            x = P[:, k] + _mv(R[:, k], self.c_pos.expand(N, -1, -1)) - torch.stack([0 * self.c_rad, 0 * self.c_rad, self.c_rad], -1)
            v = V[:, k] + _cross(W[:, k], x - P[:, k])
            d = x[..., 2]
            on = d < 0
            n = (-self.m.ke + self.m.kd * v[..., 2]) * d
            v2 = v[..., 0] ** 2 + v[..., 1] ** 2
            vt = torch.sqrt(torch.where(v2 > 0, v2, torch.ones_like(v2))) * (v2 > 0)
            slow = self.m.kt * vt <= self.m.mu * n.abs()
            sc = torch.where(slow, torch.full_like(vt, self.m.kt), self.m.mu * n.abs() / torch.where(slow, torch.ones_like(vt), vt))
            f = torch.stack([-sc * v[..., 0], -sc * v[..., 1], n], -1) * on[..., None]
            ff = ff.index_add(1, k, f)
            fn = fn.index_add(1, k, _cross(x - C[:, k], f))
        if len(self.seg):
            x = P[:, self.v_link] + _mv(R[:, self.v_link], self.v_pos.expand(N, -1, -1))
            dv = x[:, self.seg + 1] - x[:, self.seg]
            F = (a[:, self.m.n_tact:].clamp(0, 1) * self.fmax)[:, self.seg_mus, None] * dv / dv.norm(dim=-1, keepdim=True)
            for e, f in ((self.seg, F), (self.seg + 1, -F)):
                k = self.v_link[e]
                ff = ff.index_add(1, k, f)
                fn = fn.index_add(1, k, _cross(x[:, e] - C[:, k], f))
        # Jacobians of the centres of mass [N, L, nv, 3]
        sp, mv = self.spin[:, None], self.moves[..., None]
        Jw = (ax * sp).unsqueeze(1) * mv
        Jv = torch.where(sp > 0, _cross(ax.unsqueeze(1).expand(N, self.L, -1, -1), C.unsqueeze(2) - org.unsqueeze(1)), ax.unsqueeze(1)) * mv
        IJ = Jw @ Iw                                                       # Iw symmetric
        flat = lambda J: J.transpose(2, 3).flatten(1, 2)                   # noqa: E731   [N, 3 L, nv]
        Jwf, Jvf = flat(Jw), flat(Jv)
        M = flat(IJ).transpose(1, 2) @ Jwf + (flat(Jv * self.mass[:, None, None])).transpose(1, 2) @ Jvf
        f_in = self.mass[:, None] * (Ac - self.grav) - ff
        n_in = _mv(Iw, AW) + _cross(W, _mv(Iw, W)) - fn
        bias = (Jwf.transpose(1, 2) @ n_in.flatten(1).unsqueeze(-1) + Jvf.transpose(1, 2) @ f_in.flatten(1).unsqueeze(-1)).squeeze(-1)
        tau = -self.damp * qd
        if self.m.n_tact:
            tau = tau + a[:, :self.m.n_tact] @ self.gear
        if self.m.k_limit and self.limited:
            d, s = (list(x) for x in zip(*self.limited))
            x = q[:, s]
            over = (self.lo[d] - x).clamp(min=0) + (self.hi[d] - x).clamp(max=0)
            tau = tau.index_add(1, torch.tensor(d, device=q.device), self.m.k_limit * over)
        Lc = torch.linalg.cholesky(M + torch.diag(self.arm))
        return torch.cholesky_solve((tau - bias).unsqueeze(-1), Lc).squeeze(-1), R

    def substep(self, q, qd, a):
        acc, R = self.accel(q, qd, a)
        h = self.h
        qd = qd + h * acc
        if self.jt[0] != 0:
            parts = []
            for i, j in enumerate(self.jt):
                if j in (1, 2):
                    parts.append(q[:, int(self.qs[i])] + h * qd[:, int(self.ds[i])])
            return torch.stack(parts, 1), qd
        p = q[:, :3] + h * _mv(R[:, 0], qd[:, 3:6])
        u, w, om = q[:, 3:6], q[:, 6:7], qd[:, :3]
        n = torch.cat([u + 0.5 * h * (w * om + _cross(u, om)), w - 0.5 * h * (u * om).sum(-1, keepdim=True)], -1)
        return torch.cat([p, n / n.norm(dim=-1, keepdim=True), q[:, 7:] + h * qd[:, 6:]], -1), qd

    def reward(self, q, qd, a):
        c, m = self.rc, self.m
        r = -(self.rwq * q * q).sum(-1) - (self.rwqd * qd * qd).sum(-1) - c[0] * (a * a).sum(-1)
        hq = m.height_q
        if self.jt[0] == 0:
            R = _rot(*q[:, 3:7].unbind(-1))
            r = r + c[1] * _mv(R, qd[:, 3:6])[:, 0] + c[2] * R[:, 2, 2] + c[3] * R[:, 0, 0]
            hq = 2
        elif m.vx_dof >= 0:
            r = r + c[1] * qd[:, m.vx_dof]
        if hq >= 0:
            D = (q[:, hq] - c[4]).clamp(c[5], c[6])
            r = r + torch.where(D < 0, c[7] * D * D + c[8] * D, c[9] * D)
        return r

    def step(self, q, qd, a):
        """q [nq, N], qd [nv, N], a [na, N] -> post-step state and reward [N]."""
        q, qd, a = q.T, qd.T, a.T
        for _ in range(self.m.substeps):
            q, qd = self.substep(q, qd, a)
        return q.T, qd.T, self.reward(q, qd, a)


def _join(parts):
    return torch.cat([p.flatten(-2) for p in parts], -1)


def _window64(sim, q, qd, act, reset=None):
    """q_traj, qd_traj, reward (and done, episode steps) of one group; a step is recomputed in its backward."""
    qs, qds, rs, done = [q], [qd], [], []
    ep = None if reset is None else reset[2].clone()
    for t in range(act.shape[0]):
        need = torch.is_grad_enabled()
        q, qd, r = checkpoint(sim.step, q, qd, act[t], use_reentrant=False) if need else sim.step(q, qd, act[t])
        if reset is not None:
            hq = 2 if sim.jt[0] == 0 else sim.m.height_q
            ep = ep + 1
            d = (ep >= HORIZON) | (q[hq] < reset[3])
            ep = torch.where(d, torch.zeros_like(ep), ep)
            q, qd = torch.where(d, reset[0], q), torch.where(d, reset[1], qd)
            done.append(d.to(torch.uint8))
        qs.append(q)
        qds.append(qd)
        rs.append(r)
    return torch.stack(qs), torch.stack(qds), torch.stack(rs), done, ep


def _observe(q, qd):
    R = _rot(*q[3:7].unbind(0))
    v, w = _mv(R, qd[3:6].T), _mv(R, qd[0:3].T)
    return torch.cat([q[2:3], q[3:7], v.T, w.T, q[7:], qd[6:], R[:, 2, 2][None], R[:, 0, 0][None]]).T


def exact(case, seed):
    dev, kind = "cuda", case["kind"]
    if kind == "td":
        r, v, d = _td_arrays(case, seed)
        r, v = r.double(), v.double()
        gamma, lam = float(np.float32(GAMMA)), float(np.float32(LAMBDA))
        g, out = v[-1], []
        for t in range(case["h"] - 1, -1, -1):
            nxt = gamma * ((1 - lam) * v[t + 1] + lam * g)
            g = r[t] + (nxt if d is None else torch.where(d[t].bool(), torch.zeros_like(nxt), nxt))
            out.append(g)
        return torch.stack(out[::-1])
    groups, arrays, rb = _arrays(case, seed)
    t64 = lambda x: torch.tensor(np.asarray(x, np.float64), device=dev)  # noqa: E731
    rb, h, back = t64(rb), case["h"], kind not in ("step", "rollout")
    if kind == "policy":
        (m, n), (q, qd) = groups[0], (t64(x) for x in arrays[0][:2])
        sim, net = Sim64(m, dev), _policy(case, groups[0][0], seed).double()
        total = 0.0
        for _ in range(h):
            x = _observe(q, qd)
            for k, lin in enumerate(net.layers):
                x = lin(x)
                x = torch.nn.functional.elu(x) if k + 1 < len(net.layers) else torch.sigmoid(x)
            q, qd, r = checkpoint(sim.step, q, qd, x.T, use_reentrant=False)
            total = total + r.sum()
        loss = -total / (n * h)
        return [loss.detach(), *torch.autograd.grad(loss, list(net.parameters()))]
    outs, env = [], 0
    for (m, n), (q, qd, act, gq, gqd) in zip(groups, arrays):
        sim = Sim64(m, dev)
        x = [t64(y).requires_grad_(back) for y in (q, qd, act)]
        reset = None
        if kind == "episodic":
            qr, qdr, ep = _reset_arrays(case, seed, m, n)
            reset = (t64(qr), t64(qdr), torch.from_numpy(ep).to(dev), inputs.episode_rule(m)[0])
        qs, qds, rs, done, ep = _window64(sim, *x, reset)
        grads = []
        if back:
            loss = (qs[-1] * t64(gq)).sum() + (qds[-1] * t64(gqd)).sum() + (rs * rb[:, env:env + n]).sum()
            grads = [g.detach() for g in torch.autograd.grad(loss, x)]
        outs.append(([qs.detach(), qds.detach(), rs.detach()], grads, done, ep))
        env += n
    if kind == "step":
        (qs, qds, rs), = (o[0] for o in outs)
        return [qs[1].flatten(), qds[1].flatten(), rs[0]]
    f = [_join([o[0][k] for o in outs]) for k in (0, 1)] + [torch.cat([o[0][2] for o in outs], -1)]
    if kind == "autograd":
        f = [f[0][1], f[1][1], f[2][0]]
    if kind == "rollout":
        return f
    g = [_join([o[1][k] for o in outs]) for k in (0, 1, 2)]
    if kind == "episodic":
        return [*f, torch.stack(outs[0][2]), *g, outs[0][3]]
    return [*f, *g]
