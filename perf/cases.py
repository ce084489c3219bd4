"""The framework's work, as its users have it done: batched differentiable rollouts of the
workloads, system identification, policy runs, camera frames and the warm-start network's training.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same ranges, ``prepare`` makes
what a program holds before the call (models, weights, worlds, device buffers), ``run`` is one pass
through the public entry points, ``work`` what a pass cannot do without, and ``exact`` the same
pass in 64 bits, in plain torch, where that takes seconds.
"""
import math

import numpy as np
import torch

from paper_1611_01652_gb300 import binding as DP
from paper_1611_01652_gb300 import workloads as WL
from paper_1611_01652_gb300.batching import UnevenBatch

DEV = "cuda"
ALPHA = 0.7  # weight of the previous step's impulses in the damped warm start
SIZES = {"ball": (1, 0, 3), "pendulum": (3, 3, 15), "masses": (3, 3, 15), "quadruped": (9, 8, 80), "policy": (9, 8, 80)}


def listed():
    return [
        # one throw, as an interactive program simulates and differentiates it: latency alone
        dict(name="ball_one", kind="ball", batch=1, horizon=300, sweeps=20),
        # a batch of throws (shooting for the launch that hits a target)
        dict(name="ball_batch", kind="ball", batch=4096, horizon=300, sweeps=20),
        # chains over many small steps, states checkpointed every 32 steps and segments recomputed
        dict(name="pendulum_segments", kind="pendulum", batch=1024, horizon=250, sweeps=10, segment=32),
        # one iteration of the link-mass fit: parameters in, rollout, mass gradients, Adam
        dict(name="masses_fit", kind="masses", batch=4096, horizon=300, sweeps=10),
        # the learning batch of the paper (128 robots): a policy run without gradients
        dict(name="policy_128", kind="policy", batch=128, horizon=60, sweeps=10, warm=True, recurrent=0),
        # gait training: the plain solver, and the damped warm start over the full horizon
        dict(name="quadruped_plain", kind="quadruped", batch=4096, horizon=100, sweeps=20, warm=False, recurrent=0),
        dict(name="quadruped_warm", kind="quadruped", batch=4096, horizon=1000, sweeps=10, warm=True, recurrent=0),
        # a recurrent controller, ragged batch
        dict(name="quadruped_recurrent", kind="quadruped", batch=1500, horizon=100, sweeps=14, warm=True, recurrent=8),
        # the 1.1 M-parameter controller between step launches
        dict(name="quadruped_wide", kind="wide", batch=2048, horizon=50, sweeps=10, warm=True),
        # arms of 3 to 7 links with horizons of 200 to 2000 steps, one captured pass
        dict(name="arms_uneven", kind="arms", batch=2048, hmin=200, hmax=2000, sweeps=10),
        # a camera in the loop: frames and the gradient to the poses and textures
        dict(name="camera_mixed", kind="camera", batch=512, width=288, height=96, mixed=True),
        # one step of the warm-start network's training
        dict(name="warmstart_train", kind="wstrain", rows=32768),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ball", "pendulum", "masses", "policy", "quadruped", "quadruped", "wide", "arms", "camera", "wstrain"])
    if kind == "ball":
        return dict(kind=kind, batch=_logint(rng, 1, 4096), horizon=_logint(rng, 30, 300), sweeps=rng.choice([10, 20]))
    if kind == "pendulum":
        return dict(kind=kind, batch=_logint(rng, 16, 2048), horizon=_logint(rng, 50, 400), sweeps=10,
                    segment=rng.choice([0, 16, 32]))
    if kind == "masses":
        return dict(kind=kind, batch=4 * _logint(rng, 8, 1024), horizon=_logint(rng, 50, 300), sweeps=10)
    if kind == "policy":
        return dict(kind=kind, batch=_logint(rng, 1, 4096), horizon=_logint(rng, 10, 200), sweeps=rng.choice([5, 10, 20]),
                    warm=rng.random() < 0.5, recurrent=rng.choice([0, 8]))
    if kind == "quadruped":
        return dict(kind=kind, batch=_logint(rng, 16, 4096), horizon=_logint(rng, 10, 100),
                    sweeps=rng.choice([5, 7, 10, 14, 20]), warm=rng.random() < 0.5, recurrent=rng.choice([0, 0, 4, 8]))
    if kind == "wide":
        return dict(kind=kind, batch=_logint(rng, 64, 2048), horizon=_logint(rng, 10, 50), sweeps=rng.choice([5, 10, 14]),
                    warm=rng.random() < 0.5)
    if kind == "arms":
        hmax = _logint(rng, 200, 2000)
        return dict(kind=kind, batch=_logint(rng, 64, 2048), hmin=hmax // 10, hmax=hmax, sweeps=10)
    if kind == "camera":
        # even heights: on odd ones pixel centres lie exactly on the ground texture's seams
        w = rng.choice([32, 64, 144, 288])
        return dict(kind=kind, batch=_logint(rng, 4, 512), width=w, height=w // 2 + 2 * rng.randint(0, 7) if w < 288 else 96,
                    mixed=rng.random() < 0.5)
    return dict(kind=kind, rows=_logint(rng, 256, 65536))


# ------------------------------------------------------------------------------ inputs
def _tiled(base, B, rng, moving):
    """``base``'s robots repeated to a batch of B, each with masses and speeds of its own."""
    m = base.subset(np.arange(B) % base.B)
    k = rng.uniform(0.9, 1.1, size=B)
    m.mass = WL.f32(m.mass * k[:, None])
    m.inertia = WL.f32(m.inertia * k[:, None, None])
    if moving:
        m.state0[:, :, 12:14] += rng.uniform(-0.1, 0.1, size=(B, 1, 2))
        m.state0 = WL.f32(m.state0)
    return m


def _model(case, seed):
    rng = np.random.default_rng(seed)
    kind, B = case["kind"], case.get("batch")
    few = min(B, 64) if B else 0
    if kind == "ball":
        m = _tiled(WL.ball(few, seed, case["horizon"], case["sweeps"]), B, rng, True)
        m.loss_target[:, :2] = WL.f32(rng.uniform(-5, 5, size=(B, 2)))
        return m
    if kind == "pendulum":
        return _tiled(WL.pendulum3(few, seed, case["horizon"], case["sweeps"], ckpt_every=case["segment"]), B, rng, False)
    if kind == "masses":
        m = WL.pendulum_sysid(min(B, 64), 4, seed, case["horizon"], case["sweeps"])
        m = m.subset(np.arange(B) % m.B)
        m.mass = WL.f32(np.repeat(rng.uniform(0.6, 1.8, size=(B // 4, 3)), 4, axis=0))
        m.loss_target = WL.f32(rng.uniform(-1, 1, size=(B, 3)) * [1.0, 0.01, 0.2] + [0.0, 0.0, -1.0])
        return m
    if kind == "wide":
        return _tiled(WL.quadruped(few, seed, case["horizon"], case["sweeps"], widths=[64, 1024, 1024, 8]), B, rng, True)
    return _tiled(WL.quadruped(few, seed, case["horizon"], case["sweeps"], n_recurrent=case["recurrent"]), B, rng, True)


def _arms(case, seed):
    """Bins of arms by link count (uneven sizes): a few robots of each repeated, horizons drawn per
    robot."""
    rng = np.random.default_rng(seed)
    few = WL.arms(160, seed, case["sweeps"], hmin=case["hmin"], hmax=case["hmax"])
    bins = {}
    for k, n in enumerate(sorted(few)):
        c = case["batch"] * (k + 8) // 50
        m = _tiled(few[n], c, rng, False)
        m.horizons = rng.integers(case["hmin"], case["hmax"] + 1, size=c).astype(np.int32)
        m.horizon = int(m.horizons.max())
        bins[n] = m
    return bins


def _scene(case, seed):
    few = WL.camera_scene(min(case["batch"], 16), case["width"], case["height"], seed, mixed=case["mixed"])
    few.states = np.ascontiguousarray(few.states[np.arange(case["batch"]) % len(few.states)])
    return few


def _rows(case, seed):
    """Harvested rows (16 features, 3 targets) of the scales the rollouts give."""
    rng = np.random.default_rng(seed)
    x = rng.normal(size=(case["rows"], DP.WS_ROW)).astype(np.float32)
    x[:, 6:9] = np.abs(x[:, 6:9])
    x[:, 15] = rng.integers(0, 4, size=case["rows"])
    return x


def _ws_weights(seed):
    rng = np.random.default_rng(seed + 1)
    return WL.xavier_weights([16, 64, 64, 3], 0, rng)


class State:
    pass


def _dev(x):
    return torch.tensor(np.asarray(x, np.float32), device=DEV)


def prepare(case, seed):
    s = State()
    s.kind = kind = case["kind"]
    if kind == "arms":
        bins = _arms(case, seed)
        s.batch = UnevenBatch(bins, _dev(bins[min(bins)].W), tune=False)
        s.batch.capture()
        return s
    if kind == "camera":
        cs = _scene(case, seed)
        s.rig = DP.CameraRig(cs)
        s.x, s.tex = _dev(cs.states), _dev(cs.textures)
        s.image = torch.empty(case["batch"], case["height"], case["width"], 3, device=DEV)
        g = torch.Generator(DEV).manual_seed(seed)
        s.dimage = torch.randn(s.image.shape, device=DEV, generator=g) / s.image[0].numel()
        s.dx, s.dtex = torch.empty_like(s.x), torch.empty_like(s.tex)
        return s
    if kind == "wstrain":
        s.rows = _dev(_rows(case, seed))
        s.W = _dev(_ws_weights(seed))
        s.m, s.v, s.dW = (torch.zeros_like(s.W) for _ in range(3))
        s.loss = torch.zeros(1, device=DEV)
        s.work = DP.ws_workspace(case["rows"])
        s.start = s.W.clone()
        return s
    m = _model(case, seed)
    s.world = DP.World(m, warmstart=case.get("warm", False))
    if case.get("warm"):
        s.world.set_warmstart(torch.zeros(DP.WS_PARAMS, device=DEV), ALPHA)
    s.W = _dev(m.W) if m.W is not None else None
    s.x0 = _dev(m.state0)
    s.steps = case["horizon"]
    s.loss = torch.empty(m.B, device=DEV)
    s.dloss = torch.full((m.B,), 1.0 / m.B, device=DEV)
    s.x = torch.empty(m.B, m.nb, 18, device=DEV)
    s.dx = torch.empty_like(s.x)
    s.dW = torch.empty(s.world.n_params, device=DEV) if s.world.n_params else None
    if kind == "masses":
        # one value per pendulum, shared by its four swings
        s.mass = _dev(m.mass[::4])
        s.start = s.mass.clone()
        s.m, s.v, s.sum = (torch.zeros_like(s.mass) for _ in range(3))
        s.inst, s.g = _dev(m.mass), torch.zeros(m.B, 3, device=DEV)
    return s


# ------------------------------------------------------------------------------ one pass
def run(s):
    if s.kind == "arms":
        s.batch.run()
        return {"dW": s.batch.dW, "loss": [s.batch.loss[k] for k in s.batch.keys]}
    if s.kind == "camera":
        s.rig.render(s.x, s.tex, s.image)
        s.rig.render_backward(s.x, s.tex, s.dimage, s.dx, s.dtex)
        return {"image": s.image, "dstate": s.dx, "dtextures": s.dtex}
    if s.kind == "wstrain":
        s.W.copy_(s.start)
        s.m.zero_()
        s.v.zero_()
        DP.ws_loss_grad(s.W, s.rows, s.loss, s.dW, s.work)
        DP.ws_adam(s.W, s.dW, s.m, s.v, 1, 3e-3)
        return {"loss": s.loss, "dW": s.dW, "W": s.W, "m": s.m, "v": s.v}
    w = s.world
    if s.kind == "policy":
        w.set_state(s.x0)
        w.step(s.steps, s.W)
        return {"state": w.get_state(s.x)}
    if s.kind == "masses":
        s.mass.copy_(s.start)
        s.m.zero_()
        s.v.zero_()
        s.inst.view(-1, 4, 3).copy_(s.mass.unsqueeze(1))
        w.set_params(mass=s.inst)
        w.rollout(None, s.loss)
        w.backward(s.dloss, None, None, {"mass": s.g})
        torch.sum(s.g.view(-1, 4, 3), 1, out=s.sum)
        DP.ws_adam(s.mass, s.sum, s.m, s.v, 1, 0.03)
        return {"loss": s.loss, "dmass": s.g, "mass": s.mass, "state": w.get_state(s.x)}
    w.rollout(s.W, s.loss)
    w.backward(s.dloss, s.dW, s.dx)
    return {"loss": s.loss, "dW": s.dW, "dstate0": s.dx, "state": w.get_state(s.x)}


# ------------------------------------------------------------------------------ what a pass needs
def work(case):
    """Bytes: parameters, initial states and weights read once, losses, gradients and final states
    written once. Operations: the counts per instance-step of an operator-counting run of the
    engine (tests/golden), linear in the sweeps; 2 per multiply-add of the dense layers."""
    kind = case["kind"]
    if kind == "camera":
        pix, n = case["batch"] * case["width"] * case["height"], 6 if case["mixed"] else 4
        return {"bytes": pix * 24 + case["batch"] * 3 * 18 * 8, "flops": pix * (60.0 * n + 120.0)}
    if kind == "wstrain":
        return {"bytes": case["rows"] * 19 * 4 + 5443 * 32, "flops": case["rows"] * 5312 * 6.0}
    B = case["batch"]
    if kind == "arms":
        steps, nb, nj, rows = B * 0.5 * (case["hmin"] + case["hmax"]), 5, 5, 37
        net, params, back = 32 * 256 + 256 * 256 + 256 * 7, 76039, True
    else:
        nb, nj, rows = SIZES["quadruped" if kind == "wide" else kind]
        steps, back = B * case["horizon"], kind != "policy"
        net, params = 0, 0
        if kind in ("quadruped", "policy"):
            h = case["recurrent"]
            net, params = (24 + h) * 128 + 128 * 128 + 128 * (8 + h), 17544 + 256 * h
        elif kind == "wide":
            net, params = 64 * 1024 + 1024 * 1024 + 1024 * 8, 1124360
    per = rows * (145.0 + 57.4 * case["sweeps"]) + 2.0 * net
    if back:
        per += rows * (770.0 + 211.0 * case["sweeps"]) + 4.0 * net
    state = 18 * nb
    prm = 4 * nb + 23 * nj + 12 + 6 * (8 if nb == 9 else 1)
    byt = 4.0 * (B * (prm + state * (3 if back else 2) + 2) + params * (2 if back else 1))
    return {"bytes": byt, "flops": steps * per}


# ------------------------------------------------------------------------------ the same in 64 bits
MOST_ROWS = 40000  # row updates one after the other (steps x sweeps x rows) that take some ten seconds


def exact(case, seed):
    kind = case["kind"]
    if kind == "camera":
        return _exact_camera(case, seed)
    if kind == "wstrain":
        return _exact_train(case, seed)
    if kind in ("arms", "wide"):
        return None
    back = kind != "policy"
    if case["horizon"] * case["sweeps"] * SIZES[kind][2] > (MOST_ROWS if back else 2 * MOST_ROWS):
        return None
    # a bfloat16 rounding of the controller that falls the other way in 32 bits is a contact more or
    # less some steps later: beyond that the gradients in 64 bits are another robot's
    if kind == "quadruped" and case["horizon"] > 16:
        return None
    m = _model(case, seed)
    r = Engine(m, case).run(back, kind == "masses")
    if kind == "policy":
        return {"state": r["state"]}
    if kind == "masses":
        g = r["dmass"]
        sm = g.reshape(-1, 4, 3).sum(1)
        mass = torch.tensor(m.mass[::4], dtype=torch.float64)
        mom, var = 0.1 * sm, 0.001 * sm * sm
        new = mass - 0.03 * (mom / 0.1) / (torch.sqrt(var / 0.001) + 1e-8)
        return {"loss": r["loss"], "dmass": g, "mass": new, "state": r["state"]}
    return {"loss": r["loss"], "dW": r["dW"], "dstate0": r["dstate0"], "state": r["state"]}


def _bf16(x):
    """bfloat16 storage, straight through in reverse mode."""
    return x + (x.detach().to(torch.bfloat16).to(x.dtype) - x.detach())


def _mv(R, x):
    return torch.einsum("bij,bj->bi", R, x)


def _cross(a, b):
    return torch.linalg.cross(a, b)


class Engine:
    """The engine in 64 bits over a batch: contact rows, hinges, limits and servos, projected
    Gauss-Seidel in (colour, slot) order, semi-implicit Euler with R <- (3R - R R^T R) / 2, and
    reverse mode by torch's autograd."""

    def __init__(self, m, case):
        big = m.B * case["horizon"] * case["sweeps"] > 2e6
        self.dev = torch.device(DEV if big else "cpu")
        self.m, self.warm = m, case.get("warm", False)
        for k in WL.PER_INSTANCE:
            setattr(self, k, torch.tensor(getattr(m, k), dtype=torch.float64, device=self.dev))
        self.n_rec = int(getattr(m, "n_recurrent", 0))
        s = []  # slots: kind, index, sub-row, parent, child, slot of the contact's normal
        for j in range(m.nj):
            a, b = (int(x) for x in m.joint_body[j])
            s += [("lin", j, k, a, b, -1) for k in range(3)] + [("ang", j, k, a, b, -1) for k in range(2)]
        for flag, kind in ((WL.FLAG_LIMIT, "limit"), (WL.FLAG_MOTOR, "motor")):
            s += [(kind, j, 0, int(m.joint_body[j, 0]), int(m.joint_body[j, 1]), -1) for j in range(m.nj)
                  if m.joint_flags[j] & flag]
        for q in range(m.ns):
            n = len(s)
            s += [("normal", q, 0, int(m.sphere_body[q]), -1, -1)]
            s += [("friction", q, k, int(m.sphere_body[q]), -1, n) for k in range(2)]
        colour = []
        for i, x in enumerate(s):
            mine = {b for b in x[3:5] if b >= 0}
            used = {colour[k] for k in range(i) if mine & set(s[k][3:5])}
            colour.append(next(c for c in range(i + 1) if c not in used))
        self.slots, self.order = s, sorted(range(len(s)), key=lambda i: (colour[i], i))
        self.motors = [j for j in range(m.nj) if m.joint_flags[j] & WL.FLAG_MOTOR]

    def controller(self, W, x, th, thd, t, h):
        m, B = self.m, self.m.B
        f = []
        if m.features & WL.F_ANGLES:
            f += [th[j] for j in self.motors]
        if m.features & WL.F_RATES:
            f += [thd[j] for j in self.motors]
        if m.features & WL.F_CLOCK:
            ph = 2.0 * math.pi * float(np.float32(m.clock_hz)) * (t * float(np.float32(m.dt)))
            f += [torch.full((B,), v, dtype=torch.float64, device=self.dev) for v in (math.sin(ph), math.cos(ph))]
        if m.features & WL.F_IMU:
            R = x[m.imu_body][1]
            g = -R[:, 2, :]
            w = torch.einsum("bij,bi->bj", R, x[m.imu_body][3])
            f += [g[:, k] for k in range(3)] + [w[:, k] for k in range(3)]
        z = torch.stack(f, 1)
        if h is not None:
            z = torch.cat([z, h], 1)
        z = _bf16(z)
        o = 0
        for l in range(len(m.widths) - 1):
            ni, no = m.widths[l], m.widths[l + 1]
            w, b = W[o:o + ni * no].reshape(no, ni), W[o + ni * no:o + ni * no + no]
            o += ni * no + no
            z = z @ _bf16(w).T + b
            if l < len(m.widths) - 2:
                z = _bf16(torch.relu(z))
        return z

    def step(self, x, t, lam_prev, h, W, mass):
        m, dt = self.m, float(np.float32(self.m.dt))
        bh, slop = float(np.float32(m.beta)) / dt, float(np.float32(m.slop))
        dtype = dict(dtype=torch.float64, device=self.dev)
        zero3 = torch.zeros(m.B, 3, **dtype)
        eye = torch.eye(3, **dtype).expand(m.B, 3, 3)
        P = lambda b: x[b][0] if b >= 0 else zero3  # noqa: E731
        R = lambda b: x[b][1] if b >= 0 else eye  # noqa: E731
        Wv = lambda b: x[b][3] if b >= 0 else zero3  # noqa: E731
        ua, th, thd = [], [], []
        for j in range(m.nj):
            a, b = (int(v) for v in m.joint_body[j])
            u = _mv(R(a), self.axis[:, j, 0])
            wa, wb = _mv(R(a), self.ref[:, j, 0]), _mv(R(b), self.ref[:, j, 1])
            ua.append(u)
            th.append(torch.atan2((_cross(wa, wb) * u).sum(1), (wa * wb).sum(1)))
            thd.append((u * (Wv(b) - Wv(a))).sum(1))
        out = self.controller(W, x, th, thd, t, h) if W is not None else None
        if self.n_rec:
            h = torch.tanh(out[:, -self.n_rec:])
        target = {}
        for k, j in enumerate(self.motors):
            vmax = self.motor[:, j, 2]
            target[j] = torch.minimum(torch.maximum(self.motor[:, j, 0] * (out[:, k] - th[j]), -vmax), vmax)
        g = torch.tensor([float(np.float32(v)) for v in m.gravity], **dtype)
        V, im, ii = [], [], []
        for b in range(m.nb):
            Rb, I = x[b][1], self.inertia[:, b]
            Iw = torch.einsum("bik,bk,bjk->bij", Rb, I, Rb)
            Ii = torch.einsum("bik,bk,bjk->bij", Rb, 1.0 / I, Rb)
            w = x[b][3]
            w = w + dt * _mv(Ii, -_cross(w, _mv(Iw, w)))
            V.append(torch.cat([x[b][2] + dt * g, w], 1))
            im.append(1.0 / mass[:, b])
            ii.append(Ii)
        # rows: Jacobians [B, 6] per side, M^-1 J^T, effective mass, bias, bound, activity
        rows = []
        e3 = torch.eye(3, **dtype)
        for kind, i, sub, a, b, _ in self.slots:
            lin = angA = angB = zero3
            bias, bnd, on = torch.zeros(m.B, **dtype), None, torch.ones(m.B, dtype=torch.bool, device=self.dev)
            if kind == "lin":
                ra = _mv(R(a), self.anchor[:, i, 0])
                rb = _mv(R(b), self.anchor[:, i, 1])
                lin = e3[sub].expand(m.B, 3)
                angA, angB = _cross(ra, lin), -_cross(rb, lin)
                bias = bh * ((P(a) + ra) - (P(b) + rb))[:, sub]
            elif kind == "ang":
                n = self.axis[:, i, 0]
                s = torch.where(n[:, 2] >= 0, 1.0, -1.0)
                c = -1.0 / (s + n[:, 2])
                d = n[:, 0] * n[:, 1] * c
                tau = (torch.stack([1 + s * n[:, 0] ** 2 * c, s * d, -s * n[:, 0]], 1) if sub == 0 else
                       torch.stack([d, s + n[:, 1] ** 2 * c, -n[:, 1]], 1))
                angA = _mv(R(a), tau)
                angB = -angA
                bias = bh * (angA * _cross(_mv(R(b), self.axis[:, i, 1]), ua[i])).sum(1)
            elif kind == "limit":
                lo, hi = self.limit[:, i, 0], self.limit[:, i, 1]
                low, on = th[i] <= lo, (th[i] <= lo) | (th[i] >= hi)
                angB = torch.where(low, 1.0, -1.0)[:, None] * ua[i]
                angA = -angB
                bias = bh * torch.where(low, th[i] - lo, hi - th[i])
            elif kind == "motor":
                angA, angB, bias, bnd = -ua[i], ua[i], -target[i], self.motor[:, i, 1] * dt
            else:
                c = _mv(R(a), self.sph_off[:, i])
                d = (P(a) + c)[:, 2] - self.sph_rad[:, i] - float(np.float32(m.ground_z))
                on = d <= 0
                lin = e3[2 if kind == "normal" else sub].expand(m.B, 3)
                angA = _cross(c - self.sph_rad[:, i, None] * e3[2], lin)
                if kind == "normal":
                    vn = (lin * V[a][:, :3]).sum(1) + (angA * V[a][:, 3:]).sum(1)
                    bias = bh * torch.clamp(d + slop, max=0.0) + self.sph_e[:, i] * torch.clamp(vn, max=0.0)
                else:
                    bnd = self.sph_mu[:, i]
            if not bool(on.any()):
                rows.append(None)
                continue
            JA = MA = JB = MB = None
            K = 0.0
            if a >= 0:
                JA = torch.cat([lin, angA], 1)
                MA = torch.cat([im[a][:, None] * lin, _mv(ii[a], angA)], 1)
                K = K + (JA * MA).sum(1)
            if b >= 0:
                JB = torch.cat([-lin, angB], 1)
                MB = torch.cat([-im[b][:, None] * lin, _mv(ii[b], angB)], 1)
                K = K + (JB * MB).sum(1)
            meff = torch.where(on, 1.0 / (K + float(np.float32(m.gamma))), 0.0)
            rows.append((JA, JB, MA, MB, meff, torch.where(on, bias, 0.0), bnd, on))
        # start: cold, or the damped previous impulses projected on the rows' bounds (constants)
        lam = [torch.zeros(m.B, **dtype) for _ in self.slots]
        if self.warm:
            with torch.no_grad():
                for s, (kind, _, _, _, _, nrm) in enumerate(self.slots):
                    if rows[s] is None or kind == "limit":
                        continue
                    v = torch.where(rows[s][7], float(np.float32(ALPHA)) * lam_prev[s], 0.0)
                    if kind == "normal":
                        v = v.clamp(min=0.0)
                    elif kind in ("motor", "friction"):
                        hi = rows[s][6] if kind == "motor" else rows[s][6] * lam[nrm]
                        v = torch.minimum(torch.maximum(v, -hi), hi)
                    lam[s] = v
            for s, (_, _, _, a, b, _) in enumerate(self.slots):
                if rows[s] is not None:
                    if a >= 0:
                        V[a] = V[a] + lam[s][:, None] * rows[s][2]
                    if b >= 0:
                        V[b] = V[b] + lam[s][:, None] * rows[s][3]
        for _ in range(m.iters):
            for s in self.order:
                if rows[s] is None:
                    continue
                kind, _, _, a, b, nrm = self.slots[s]
                JA, JB, MA, MB, meff, bias, bnd, _ = rows[s]
                jv = bias
                if a >= 0:
                    jv = jv + (JA * V[a]).sum(1)
                if b >= 0:
                    jv = jv + (JB * V[b]).sum(1)
                new = lam[s] - meff * (jv + float(np.float32(m.gamma)) * lam[s])
                if kind in ("limit", "normal"):
                    new = torch.where(new < 0, torch.zeros_like(new), new)
                elif kind in ("motor", "friction"):
                    hi = bnd if kind == "motor" else bnd * lam[nrm]
                    new = torch.where(new < -hi, -hi, torch.where(new > hi, hi, new))
                dl = (new - lam[s])[:, None]
                lam[s] = new
                if a >= 0:
                    V[a] = V[a] + dl * MA
                if b >= 0:
                    V[b] = V[b] + dl * MB
        y = []
        for b in range(m.nb):
            v, w = V[b][:, :3], V[b][:, 3:]
            A = x[b][1] + dt * torch.linalg.cross(w[:, :, None].expand(m.B, 3, 3), x[b][1], dim=1)
            y.append((x[b][0] + dt * v, 0.5 * (3.0 * A - A @ (A.transpose(1, 2) @ A)), v, w))
        return y, [v.detach() for v in lam], h

    def point(self, x):
        b = self.m.loss_body
        return x[b][0] + _mv(x[b][1], self.loss_point)

    def run(self, back, by_mass):
        m = self.m
        W = torch.tensor(m.W, dtype=torch.float64, device=self.dev) if m.W is not None else None
        s0, mass = self.state0.clone(), self.mass.clone()
        want = [v for v in ([mass] if by_mass else [s0, W]) if v is not None] if back else []
        for v in want:
            v.requires_grad_(True)
        split = lambda s: [(s[:, b, 0:3], s[:, b, 3:12].reshape(m.B, 3, 3), s[:, b, 12:15], s[:, b, 15:18])  # noqa: E731
                           for b in range(m.nb)]
        with torch.set_grad_enabled(back):
            x = split(s0)
            q0 = self.point(x)
            lam = [torch.zeros(m.B, dtype=torch.float64, device=self.dev) for _ in self.slots]
            h = torch.zeros(m.B, self.n_rec, dtype=torch.float64, device=self.dev) if self.n_rec else None
            for t in range(m.horizon):
                x, lam, h = self.step(x, t, lam, h, W, mass)
            q, y = self.point(x), self.loss_target
            if m.loss_kind == WL.L_SQDIST:
                loss = ((q - y) ** 2).sum(1)
            elif m.loss_kind == WL.L_DISP:
                loss = (y * (q - q0)).sum(1)
            else:
                loss = (y * q).sum(1)
            g = torch.autograd.grad(loss.sum() / m.B, want) if back else ()
        flat = torch.stack([torch.cat([p, r.reshape(m.B, 9), v, w], 1) for p, r, v, w in x], 1)
        r = {"loss": loss.detach().cpu(), "state": flat.detach().cpu(), "dW": None}
        for k, v in zip(["dmass"] if by_mass else ["dstate0", "dW"], g):
            r[k] = v.cpu()
        return r


def _exact_train(case, seed):
    rows = torch.tensor(_rows(case, seed), dtype=torch.float64)
    W = torch.tensor(_ws_weights(seed), dtype=torch.float64, requires_grad=True)
    z, o = _bf16(rows[:, :16]), 0
    for ni, no in ((16, 64), (64, 64), (64, 3)):
        w, b = W[o:o + ni * no].reshape(no, ni), W[o + ni * no:o + ni * no + no]
        o += ni * no + no
        z = z @ _bf16(w).T + b
        if no == 64:
            z = _bf16(torch.relu(z))
    loss = ((z - rows[:, 16:]) ** 2).sum() / case["rows"]
    (g,) = torch.autograd.grad(loss, W)
    m, v = 0.1 * g, 0.001 * g * g
    new = W.detach() - 3e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return {"loss": loss.detach().reshape(1), "dW": g, "W": new, "m": m, "v": v}


def _exact_camera(case, seed):
    """Pixel-centre rays against boxes, spheres and planes, the nearest hit in front of the
    projection plane, bilinear texels; gradients to the states and texels of the hits taken."""
    cs = _scene(case, seed)
    B, W, H = case["batch"], case["width"], case["height"]
    g = torch.Generator(DEV).manual_seed(seed)
    dimage = torch.randn(B, H, W, 3, device=DEV, generator=g) / (H * W * 3)
    f64 = dict(dtype=torch.float64, device=DEV)
    c32 = lambda v: torch.tensor(np.asarray(v, np.float32), **f64)  # noqa: E731
    tex = c32(cs.textures).requires_grad_(True)
    dtex = torch.zeros_like(tex)
    image, dstate = torch.zeros(B, H, W, 3, **f64), torch.zeros(B, 3, 18, **f64)
    C, Rc, plane, f = c32(cs.cam_pos), c32(cs.cam_rot), float(np.float32(cs.plane)), float(np.float32(cs.f))
    jj, ii = torch.arange(W, **f64), torch.arange(H, **f64)
    px = torch.stack([(plane * (jj + 0.5 - 0.5 * W) / f)[None, :].expand(H, W),
                      (plane * (ii + 0.5 - 0.5 * H) / f)[:, None].expand(H, W), torch.full((H, W), plane, **f64)], -1)
    d = (px @ Rc).reshape(-1, 3)  # world ray directions, the same in every instance
    kinds = np.asarray(getattr(cs, "obj_kind", np.zeros(len(cs.obj_body))), int)
    half, cen = c32(cs.obj_half), c32(cs.obj_center)
    th, tw = cs.textures.shape[1:3]
    for i0 in range(0, B, 16):
        st = c32(cs.states[i0:i0 + 16]).requires_grad_(True)
        n = st.shape[0]
        best = torch.full((n, H * W), math.inf, **f64)
        colour = torch.zeros(n, H * W, 3, **f64)
        for o, body in enumerate(cs.obj_body):
            R = st[:, body, 3:12].reshape(n, 3, 3) if body >= 0 else torch.eye(3, **f64).expand(n, 3, 3)
            p = st[:, body, 0:3] if body >= 0 else torch.zeros(n, 3, **f64)
            ol = torch.einsum("bij,bi->bj", R, C - (p + R @ cen[o]))[:, None, :].expand(n, H * W, 3)
            dl = torch.einsum("pi,bij->bpj", d, R)
            hh = half[o]
            if kinds[o] == 0:
                dl = torch.where(dl == 0, torch.full_like(dl, 1e-30), dl)  # a ray along the slab
                near, far = (-torch.sign(dl) * hh - ol) / dl, (torch.sign(dl) * hh - ol) / dl
                t, k = near.max(-1)
                ok = t <= far.min(-1).values
                q = ol + t[..., None] * dl
                a, c = (k + 1) % 3, (k + 2) % 3
                u = 0.5 * (q.gather(-1, a[..., None])[..., 0] / hh[a] + 1)
                v = 0.5 * (q.gather(-1, c[..., None])[..., 0] / hh[c] + 1)
            elif kinds[o] == 1:
                A, b = (dl * dl).sum(-1), (dl * ol).sum(-1)
                disc = A * hh[0] ** 2 - (torch.linalg.cross(dl, ol) ** 2).sum(-1)
                ok = disc >= 0
                t = (-b - torch.sqrt(torch.where(ok, disc, torch.ones_like(disc)))) / A
                q = torch.where(ok[..., None], ol + t[..., None] * dl, torch.tensor([0.6, 0.0, 0.8], **f64) * hh[0])
                u = torch.atan2(q[..., 1], q[..., 0]) / (2 * math.pi) + 0.5
                v = torch.acos((q[..., 2] / hh[0]).clamp(-1, 1)) / math.pi
            else:
                ok = dl[..., 2] != 0
                t = -ol[..., 2] / torch.where(ok, dl[..., 2], torch.ones_like(dl[..., 2]))
                q = ol + t[..., None] * dl
                u, v = q[..., 0] / (2 * hh[0]) + 0.5, q[..., 1] / (2 * hh[1]) + 0.5
                u, v = u - u.detach().floor(), v - v.detach().floor()
            win = ok & (t >= 1) & (t < best)
            best = torch.where(win, t, best).detach()
            xs, ys = torch.where(win, u, torch.zeros_like(u)) * tw - 0.5, torch.where(win, v, torch.zeros_like(v)) * th - 0.5
            x0, y0 = xs.detach().floor(), ys.detach().floor()
            fx, fy = (xs - x0)[..., None], (ys - y0)[..., None]
            T = tex[int(cs.obj_tex[o])]
            X = [(x0.long() + e).clamp(0, tw - 1) for e in (0, 1)]
            Y = [(y0.long() + e).clamp(0, th - 1) for e in (0, 1)]
            smp = ((1 - fx) * (1 - fy) * T[Y[0], X[0]] + fx * (1 - fy) * T[Y[0], X[1]] +
                   (1 - fx) * fy * T[Y[1], X[0]] + fx * fy * T[Y[1], X[1]])
            colour = torch.where(win[..., None], smp, colour)
        gs, gt = torch.autograd.grad((colour * dimage[i0:i0 + 16].reshape(n, -1, 3)).sum(), [st, tex])
        image[i0:i0 + 16] = colour.detach().reshape(n, H, W, 3)
        dstate[i0:i0 + 16] = gs
        dtex += gt
    return {"image": image.cpu(), "dstate": dstate.cpu(), "dtextures": dtex.cpu()}
