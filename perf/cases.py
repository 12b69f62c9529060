"""Workloads the framework is timed on, with the inputs, one pass of each and its values in 64 bits.

Every case goes through the package's public entry points (``RodBatch``, the C names of
``corde`` and ``RodRollout``) the way a program that uses them does.  Sizes and materials
are those of ``paper_2509_04277_gb300.workloads`` and of the benchmark.

A case's ``kind``:

  rod      one clamped rod (``ext``: the extensible variant) driven at its base: ``calls``
           calls of ``steps`` time steps, each with its own drive sample and its own
           positions out, then the whole state;
  vessel   the same inside a curved vessel;
  knot     the same on a torus knot with self-collision;
  pair     catheter and guidewire bound in mode ``mode``, then the whole state;
  batch    ``rods`` independent rods of uneven lengths, ``steps`` steps in one call;
  grad     a training step over ``rods`` rods: rollout, tip-target loss, backward pass.

``keep``: the simulation goes on from pass to pass (a haptic loop); otherwise a pass first
sets the initial state (a what-if run, a sample, a training step).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2509_04277_gb300 import corde
from paper_2509_04277_gb300 import workloads as W
from paper_2509_04277_gb300.autograd import RodRollout

DT_TICK = 1000  # drive samples in one period of the seeded drives (one second at 1 kHz)


# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # a short extensible pendulum, one call per look at it: latency of one small launch
        {"name": "pendulum_64", "kind": "rod", "ext": True, "n": 64, "calls": 1, "steps": 10, "keep": True},
        # the headline: a 512-node guidewire at haptic rate, 16 ticks of 10 steps per frame,
        # on the kernel variant that the tuner and the benchmark give it
        {"name": "guidewire_512", "kind": "rod", "ext": False, "n": 512, "calls": 16, "steps": 10, "keep": True,
         "ept": 2, "nt": 256},
        # an odd length on the default plan, one time step per call (the tightest coupling)
        {"name": "guidewire_777_1step", "kind": "rod", "ext": False, "n": 777, "calls": 16, "steps": 1, "keep": False},
        # the longest rod of a single block
        {"name": "rod_2048", "kind": "rod", "ext": False, "n": 2048, "calls": 4, "steps": 10, "keep": False},
        # a rod over a cluster, ragged length
        {"name": "rod_5000", "kind": "rod", "ext": False, "n": 5000, "calls": 4, "steps": 10, "keep": False},
        # a rod longer than a cluster holds
        {"name": "rod_65536", "kind": "rod", "ext": False, "n": 65536, "calls": 4, "steps": 10, "keep": False},
        # insertion into a vessel
        {"name": "vessel_512", "kind": "vessel", "n": 512, "calls": 8, "steps": 10, "keep": False},
        # self-collision
        {"name": "knot_512", "kind": "knot", "n": 512, "calls": 4, "steps": 10, "keep": False},
        # catheter and guidewire with two-way binding
        {"name": "pair_512", "kind": "pair", "n": 512, "mode": 2, "calls": 8, "steps": 10, "keep": False},
        # throughput: thousands of uneven rods
        {"name": "batch_4096", "kind": "batch", "rods": 4096, "n_min": 16, "n_max": 2048, "iters": 10, "steps": 100},
        # material identification of one rod, and of many at once
        {"name": "grad_1x256", "kind": "grad", "rods": 1, "n": 256, "steps": 200, "every": 20},
        {"name": "grad_256x256", "kind": "grad", "rods": 256, "n": 256, "steps": 200, "every": 20},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    seed = {"mat": rng.randrange(1 << 20)}
    kind = rng.choice(["rod", "rod", "rod", "vessel", "knot", "pair", "batch", "grad"])
    if kind == "rod":
        ext = rng.random() < 0.25
        n = _log(rng, 8, 65536)
        return {"kind": "rod", "ext": ext, "n": n, "calls": rng.choice([1, 4, 8]), "steps": rng.choice([1, 5, 10, 20]),
                "keep": False, **seed}
    if kind == "vessel":
        return {"kind": "vessel", "n": _log(rng, 100, 512), "calls": rng.choice([1, 4, 8]), "steps": rng.choice([1, 5, 10]),
                "keep": False, **seed}
    if kind == "knot":
        return {"kind": "knot", "n": _log(rng, 128, 512), "calls": rng.choice([1, 2, 4]), "steps": rng.choice([1, 5, 10]),
                "keep": False, **seed}
    if kind == "pair":
        return {"kind": "pair", "n": _log(rng, 40, 1024), "mode": rng.randrange(3), "calls": rng.choice([1, 4, 8]),
                "steps": rng.choice([1, 5, 10]), "keep": False, **seed}
    if kind == "batch":
        return {"kind": "batch", "rods": _log(rng, 2, 2048), "n_min": 16, "n_max": rng.choice([256, 1024, 2048]),
                "iters": rng.choice([5, 10, 20]), "steps": rng.choice([10, 30, 50]), **seed}
    return {"kind": "grad", "rods": _log(rng, 1, 128), "n": _log(rng, 16, 512), "steps": rng.choice([40, 100]),
            "every": rng.choice([10, 20]), **seed}


# --------------------------------------------------------------------------- inputs


def _uneven(ns, iters, g):
    """Clamped pendulums of the given lengths, drawn like ``workloads.batched_rods``."""
    rods = len(ns)
    E, r = g.uniform(1e9, 100e9, size=rods), g.uniform(0.2e-3, 2e-3, size=rods)
    q0 = g.standard_normal((rods, 4))
    q0 /= np.linalg.norm(q0, axis=1, keepdims=True)
    out = []
    for k in range(rods):
        n, m = int(ns[k]), int(ns[k]) - 1

        def turned(sigma):
            v = g.standard_normal((m, 3)) * sigma
            return _qmul_np(q0[k][None, :], np.concatenate([v / 2, np.sqrt(1 - (v * v).sum(1, keepdims=True) / 4)], 1))

        frames, tilts = turned(1e-3), turned(1e-3)
        frames[0] = q0[k]
        x, y, z, w = tilts.T
        d3 = np.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], 1)
        pos = np.concatenate([np.zeros((1, 3)), np.cumsum(d3 / m, axis=0)])
        out.append(W.RodSpec(
            n_nodes=n, length=1.0, radius=float(r[k]), E_bend=float(E[k]), E_stretch=float(E[k]), G=float(E[k]) / 2.6,
            density=6500.0, dt=1e-4, n_iters=iters, gravity=(0.0, 0.0, -9.81), pos=pos, quat=frames,
            rest_quat=np.tile(q0[k], (m, 1)), vel=np.zeros((n, 3)), omega=np.zeros((m, 3))))
    return out


def _qmul_np(a, b):
    ax, ay, az, aw = np.moveaxis(a, -1, 0)
    bx, by, bz, bw = np.moveaxis(b, -1, 0)
    return np.stack([aw * bx + ax * bw + ay * bz - az * by, aw * by - ax * bz + ay * bw + az * bx,
                     aw * bz + ax * by - ay * bx + az * bw, aw * bw - ax * bx - ay * by - az * bz], -1)


def _inputs(case, seed):
    """Rods, drive samples [ticks, rods, 8] (None: at rest) and the kind's extra data."""
    g = W.rng(seed * 7919 + int(case.get("mat", 0)) + 11)
    kind, tick = case["kind"], 1e-4 * case["steps"]
    s = int(g.integers(1 << 30))
    if kind == "rod":
        if case["ext"]:
            return [W.extensible_pendulum(case["n"], seed=s)], None, None
        # a hand that pushes and pulls at 0.1 to 0.2 m/s and twists, one period in DT_TICK samples
        t = 2 * math.pi * np.arange(DT_TICK) / DT_TICK
        d = np.zeros((DT_TICK, 1, 8))
        d[:, 0, 0] = g.uniform(0.1, 0.2) * np.cos(t + g.uniform(-0.7, 0.7))
        d[:, 0, 6] = g.uniform(1.0, 3.0) * np.cos(t + g.uniform(-0.7, 0.7))
        return [W.guidewire(case["n"], seed=s)], d, None
    if kind == "vessel":
        rod, tube = W.vessel_guidewire(case["n"], seed=s)
        d = np.zeros((case["calls"], 1, 8))
        d[..., 0], d[..., 6] = g.uniform(0.03, 0.07), g.uniform(-2.0, 2.0)
        return [rod], d, tube
    if kind == "knot":
        d = np.zeros((case["calls"], 1, 8))
        d[..., 0], d[..., 6] = -0.05, g.uniform(1.0, 2.0)
        return [W.torus_knot(case["n"], seed=s)], d, 0.1
    if kind == "pair":
        beta0 = -(0.2 * case["n"] + float(g.uniform(0.0, 1.0)))
        cat, gw = W.catheter_guidewire(case["n"], seed=s, beta0=beta0)
        dc, dg = W.pair_drives(s, case["calls"], tick, gw.length / (case["n"] - 1), beta0)
        return [cat, gw], np.stack([dc, dg], 1), None
    if kind == "batch":
        ns = W.batched_lengths(case["rods"], 4 + int(case.get("mat", 0)), case["n_min"], case["n_max"])
        return _uneven(ns, case["iters"], g), None, None
    rods = [W.adjoint_rod(case["n"], seed=s + k) for k in range(case["rods"])]
    target = np.stack([W.tip_target(s + k, case["steps"], 1e-4, r.pos[-1]) for k, r in enumerate(rods)], 1)
    return rods, None, target


def _padded(rods):
    """Initial state as [elements, 4] float32 device tensors (frames end one element early)."""
    out = {k: [] for k in ("pos", "quat", "vel", "omega")}
    for r in rods:
        n = r.n_nodes
        q = np.zeros((n, 4))
        q[:, 3] = 1.0
        q[:n - 1] = r.quat
        out["quat"].append(q)
        for key, a in (("pos", r.pos), ("vel", r.vel), ("omega", r.omega)):
            p = np.zeros((n, 4))
            p[:len(a), :3] = a
            out[key].append(p)
    return {k: torch.tensor(np.concatenate(v), dtype=torch.float32, device="cuda") for k, v in out.items()}


def _joints(rods):
    """Per-joint stiffness and intrinsic Darboux vectors, [elements, 4] float32 each."""
    K, U = [], []
    for r in rods:
        c = _constants(r)
        n = r.n_nodes
        k, u = np.zeros((n, 4)), np.zeros((n, 4))
        k[:n - 2, :3] = [c["K1"], c["K1"], c["K3"]]
        if r.stiff_mul is not None:
            k[:n - 2, :3] *= np.asarray(r.stiff_mul, dtype=np.float32)
        a = np.asarray(r.rest_quat, dtype=np.float32).astype(np.float64)
        rel = _qmul_np(a[:-1] * np.array([-1.0, -1.0, -1.0, 1.0]), a[1:])
        u[:n - 2, :3] = 2.0 / c["l0"] * rel[:, :3]
        K.append(k)
        U.append(u)
    return tuple(torch.tensor(np.concatenate(a), dtype=torch.float32, device="cuda") for a in (K, U))


def prepare(case, seed):
    rods, drive, extra = _inputs(case, seed)
    b = corde.RodBatch(rods)
    if "ept" in case:
        b.set_plan(case["ept"], case["nt"])
    st = {"case": case, "batch": b, "at": 0, "initial": _padded(rods),
          "drive": None if drive is None else torch.tensor(drive, dtype=torch.float32, device="cuda").contiguous()}
    if case["kind"] == "vessel":
        b.set_tube(0, extra)
    elif case["kind"] == "knot":
        b.set_self_collision(0, extra)
    elif case["kind"] == "pair":
        b.bind(0, 1, case["mode"])
    elif case["kind"] == "grad":
        st["K"], st["uhat"] = _joints(rods)
        st["target"] = torch.tensor(extra, dtype=torch.float32, device="cuda")
        st["tips"] = torch.tensor(b.offsets[1:] - 1, device="cuda")
    return st


# --------------------------------------------------------------------------- one pass


def run(st):
    case, b, x0 = st["case"], st["batch"], st["initial"]
    if case["kind"] == "grad":
        leaf = {k: v.clone().requires_grad_() for k, v in
                (("K", st["K"]), ("uhat", st["uhat"]), ("vel", x0["vel"]), ("pos", x0["pos"]), ("omega", x0["omega"]))}
        traj = RodRollout.apply(b, case["steps"], case["every"], leaf["K"], leaf["uhat"], leaf["vel"], leaf["pos"],
                                x0["quat"], leaf["omega"])
        loss = (traj[:, st["tips"], :3] - st["target"]).square().sum()
        loss.backward()
        return {"loss": loss.detach(), "traj": traj.detach()[..., :3], "grad": {k: v.grad for k, v in leaf.items()}}
    if not case.get("keep"):
        corde.rod_set_state(b.handle, x0["pos"], x0["quat"], x0["vel"], x0["omega"])
    calls = case.get("calls", 1)
    out = {k: torch.empty((b.n_elem, 4), device="cuda") for k in ("pos", "quat", "vel", "omega")}
    if case["kind"] in ("rod", "vessel"):  # every call hands its positions out, as a haptic loop reads them
        ticks = torch.empty((calls, b.n_elem, 4), device="cuda")
        for k in range(calls):
            d = None if st["drive"] is None else st["drive"][(st["at"] + k) % len(st["drive"])]
            corde.rod_step_io(b.handle, case["steps"], d, ticks[k])
        corde.rod_get_state(b.handle, None, out["quat"], out["vel"], out["omega"])
        del out["pos"]
        out["ticks"], out["inv_mass"] = ticks[..., :3], ticks[..., 3]
    else:
        for k in range(calls):
            b.step(case["steps"], drive=None if st["drive"] is None else st["drive"][k])
        corde.rod_get_state(b.handle, out["pos"], out["quat"], out["vel"], out["omega"])
        out["inv_mass"] = out["pos"][:, 3]
        out["pos"] = out["pos"][:, :3]
    if case.get("keep"):
        st["at"] += calls
    return out


def work(case):
    """Floating-point operations of the time steps (elements x steps x operations of an
    element's step: 293 for the forces and the update, 41 per constraint iteration) and the
    bytes in and out: state and joint parameters once, state and positions out once."""
    kind, iters = case["kind"], case.get("iters", 10)
    calls, steps, rods = case.get("calls", 1), case["steps"], case.get("rods", 2 if kind == "pair" else 1)
    if kind == "batch":
        n = float(W.batched_lengths(rods, 4 + int(case.get("mat", 0)), case["n_min"], case["n_max"]).mean())
    else:
        n = case["n"]
    e = rods * n
    per = 306 if case.get("ext") else 293 + 41 * iters
    if kind == "grad":
        # forward, and a reverse step of about twice its operations; the trajectory written and
        # its gradient read, the leaves in and their gradients out
        return {"bytes": e * (16.0 * steps * 2 + 12 * 16), "flops": 3.0 * e * steps * per}
    return {"bytes": e * (160.0 + 16.0 * (calls if kind in ("rod", "vessel") else 0)), "flops": float(e * per * calls * steps)}


# --------------------------------------------------------------------------- 64 bits


def _constants(r):
    """Constants of one rod, from its material and the default rules for the penalty and the inertial scales."""
    l0 = r.length / (r.n_nodes - 1)
    A, I = math.pi * r.radius ** 2, math.pi * r.radius ** 4 / 4
    K1, K3, Ks = r.E_bend * I, 2 * r.G * I, r.E_stretch * A
    Kp = r.Kp if r.Kp > 0 else 400 * K1 / r.length ** 2
    m, J = r.density * A * l0, r.density * l0 * I
    ms, js = r.mass_scale, r.inertia_scale
    if not ms > 0:
        k = Kp / l0 if r.inextensible else max(Kp, Ks) / l0
        ms = max(1.0, 16 * r.dt ** 2 * k / m)
    if not js > 0:
        js = max(1.0, 4 * r.dt ** 2 * (4 * max(K1, K3) / l0 + Kp * l0) / J)
    return {"l0": l0, "K1": K1, "K3": K3, "Ks": Ks, "Kp": Kp, "ms": ms, "J1": js * J, "J3": 2 * js * J, "m": m}


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _qmul(a, b):
    av, aw, bv, bw = a[..., :3], a[..., 3:], b[..., :3], b[..., 3:]
    return torch.cat([aw * bv + bw * av + torch.linalg.cross(av, bv), aw * bw - _dot(av, bv)], -1)


class _Rods64:
    """The time step of the rods in 64 bits, all rods' elements in one array."""

    def __init__(self, rods, dev="cuda"):
        n = np.array([r.n_nodes for r in rods])
        off = np.concatenate([[0], np.cumsum(n)])
        E = int(off[-1])
        idx = np.arange(E)
        rod = np.repeat(np.arange(len(rods)), n)
        loc, last = idx - off[rod], n[rod] - 1
        c = [_constants(r) for r in rods]
        T = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        col = lambda key: T(np.array([k[key] for k in c])[rod])[:, None]  # noqa: E731
        ix = lambda mask: torch.tensor(np.nonzero(mask)[0], device=dev)  # noqa: E731
        self.E, self.dt = E, rods[0].dt
        self.l0, self.Kp, self.Ks = col("l0"), col("Kp"), col("Ks")
        self.J = torch.cat([col("J1"), col("J1"), col("J3")], 1)
        mass = np.array([k["m"] for k in c])[rod] * np.where((loc == 0) | (loc == last), 0.5, 1.0)
        w = 1.0 / (np.array([k["ms"] for k in c])[rod] * mass)
        clamp = np.array([bool(r.clamp) for r in rods])[rod] & (loc == 0)
        w[clamp] = 0.0
        self.w = T(w)[:, None]
        self.grav = T(np.array([np.array(r.gravity) / k["ms"] for r, k in zip(rods, c)])[rod]) * (self.w > 0)
        self.damp = T(np.array([1.0 / (1.0 + r.damping_alpha * r.dt) for r in rods])[rod])[:, None]
        self.bases, self.base_rod = ix(clamp), rod[clamp]
        self.seg, self.joint = ix(loc < last), ix(loc < last - 1)
        self.free_frame = T(((loc < last) & ~clamp).astype(float))[:, None]
        self.half = [ix((loc < last) & (loc % 2 == p)) for p in (0, 1)]
        self.inext, self.iters = bool(rods[0].inextensible), int(rods[0].n_iters)
        f = lambda a: T(np.asarray(a, dtype=np.float32))  # noqa: E731
        pad = lambda a, m, fill: np.concatenate([np.asarray(a), np.tile(fill, (m, 1))])  # noqa: E731
        self.x = (f(np.concatenate([r.pos for r in rods])),
                  f(np.concatenate([r.vel for r in rods])),
                  f(np.concatenate([pad(r.quat, 1, [0.0, 0.0, 0.0, 1.0]) for r in rods])),
                  f(np.concatenate([pad(r.omega, 1, [0.0, 0.0, 0.0]) for r in rods])))
        self.hook = None  # contact or binding: called with (r, v) after each iteration's sweeps
        self.before = None

    def forces(self, r, q, K, uhat):
        s, j, l0 = self.seg, self.joint, self.l0
        e = r[s + 1] - r[s]
        ln = _dot(e, e).sqrt()
        t = e / ln
        qs = q[s]
        x, y, z, w = qs.unbind(-1)
        d3 = torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], -1)
        k = l0[s] * self.Kp[s]
        f = k / ln * (d3 - _dot(t, d3) * t)
        if not self.inext:
            f = f - self.Ks[s] * (ln / l0[s] - 1) * t
        F = torch.zeros_like(r).index_add(0, s, -f).index_add(0, s + 1, f)
        con = torch.tensor([-1.0, -1.0, -1.0, 1.0], dtype=torch.float64, device=q.device)
        tb = _qmul(_qmul(qs * con, torch.cat([t, torch.zeros_like(ln)], -1)), qs)
        tq = k * torch.stack([-tb[:, 1], tb[:, 0], torch.zeros_like(tb[:, 0])], -1)
        D = _qmul(q[j] * con, q[j + 1])
        m = 2 * K[j, :3] * (2 / l0[j] * D[:, :3] - uhat[j, :3])
        c = torch.linalg.cross(D[:, :3], m)
        tau = torch.zeros_like(r).index_add(0, s, tq).index_add(0, j, 0.5 * (D[:, 3:] * m + c))
        return F, tau.index_add(0, j + 1, 0.5 * (c - D[:, 3:] * m))

    def step(self, x, K, uhat, drive):
        r, v, q, om = x
        dt = self.dt
        F, tau = self.forces(r, q, K, uhat)
        v = torch.where(self.w > 0, self.damp * (v + dt * (self.w * F + self.grav)), v)
        on = self.damp * (om + dt * (tau - torch.linalg.cross(om, self.J * om)) / self.J)
        om = torch.where(self.free_frame > 0, on, om)
        if len(self.bases):
            z = torch.zeros((len(self.bases), 3), dtype=torch.float64, device=r.device)
            v = v.index_copy(0, self.bases, z if drive is None else drive[self.base_rod, :3])
            om = om.index_copy(0, self.bases, z if drive is None else drive[self.base_rod, 4:7])
        s = self.seg
        dq = 0.5 * dt * _qmul(q[s], torch.cat([om[s], torch.zeros_like(om[s][:, :1])], -1))
        qn = q[s] + dq
        q = q.index_copy(0, s, qn / _dot(qn, qn).sqrt())
        if self.inext:
            if self.before is not None:
                self.before(r)
            half = [(a, r[a + 1] - r[a], self.w[a], self.w[a + 1]) for a in self.half]
            for _ in range(self.iters):
                for a, e, wa, wb in half:
                    d = e + dt * (v[a + 1] - v[a])
                    g = (self.l0[a] / _dot(d, d).sqrt() - 1) / (dt * (wa + wb)) * d
                    v = v.index_add(0, a, -wa * g).index_add(0, a + 1, wb * g)
                if self.hook is not None:
                    v = self.hook(r, v)
        return r + dt * v, v, q, om


def _vessel64(S, rod, tube):
    cx, cy, cz, rc, rt, mu = (float(a) for a in tube)
    allow, dt = rt - rod.radius, S.dt

    def hook(r, v):
        p = r + dt * v
        dx, dy = p[:, :1] - cx, p[:, 1:2] - cy
        rho = (dx * dx + dy * dy).sqrt()
        delta = torch.cat([dx - rc * dx / rho, dy - rc * dy / rho, p[:, 2:] - cz], -1)
        dist = _dot(delta, delta).sqrt()
        n = delta / dist
        dvn = (allow - dist) / dt
        vt = v - _dot(v, n) * n
        keep = (1 - mu * dvn.abs() / _dot(vt, vt).sqrt().clamp_min(1e-300)).clamp_min(0.0)
        return torch.where((S.w > 0) & (dist > allow), v + dvn * n - (1 - keep) * vt, v)

    S.hook = hook


def _knot64(S, rod, mu):
    two_r, sep, dt = 2 * rod.radius, max(2, int(2 * rod.radius / (rod.length / (rod.n_nodes - 1))) + 1), S.dt
    pairs = {}

    def before(r):
        i = torch.arange(S.E, device=r.device)
        near = torch.cdist(r, r, compute_mode="donot_use_mm_for_euclid_dist") < 1.5 * two_r
        pairs["ij"] = torch.nonzero(near & (i[None, :] - i[:, None] >= sep)).unbind(1)

    def hook(r, v):
        i, j = pairs["ij"]
        u = v[j] - v[i]
        delta = r[j] - r[i] + dt * u
        dist = _dot(delta, delta).sqrt()
        phi = (two_r - dist).clamp_min(0.0)
        n = delta / dist
        ut = u - _dot(u, n) * n
        cut = (mu * phi / dt / _dot(ut, ut).sqrt().clamp_min(1e-300)).clamp_max(1.0)
        J = phi * (phi / dt * n - cut * ut) / (S.w[i] + S.w[j])
        acc = torch.zeros_like(v).index_add(0, i, -J).index_add(0, j, J)
        wphi = torch.zeros_like(S.w).index_add(0, i, phi).index_add(0, j, phi)
        return torch.where(wphi > 0, v + S.w * acc / wphi.clamp_min(1e-300), v)

    S.before, S.hook = before, hook


def _pair64(S, n, mode):
    """Binding of the inner rod's nodes (elements n ..) to the outer centreline; S.beta is set per call."""
    dt = S.dt

    def hook(r, v):
        k0 = math.floor(S.beta)
        a = S.beta - k0
        for color in ((0, 1) if mode else ()):
            i = torch.arange(color, n, 2, device=r.device)
            k = i + k0
            i, k = i[(k >= 0) & (k <= n - 2)] + n, k[(k >= 0) & (k <= n - 2)]
            wk, wk1 = (S.w[k], S.w[k + 1]) if mode == 2 else (0 * S.w[k], 0 * S.w[k])
            weff = S.w[i] + (1 - a) ** 2 * wk + a * a * wk1
            d = r[i] - (1 - a) * r[k] - a * r[k + 1] + dt * (v[i] - (1 - a) * v[k] - a * v[k + 1])
            lam = torch.where(weff > 0, -d / (dt * weff.clamp_min(1e-300)), torch.zeros_like(d))
            v = v.index_add(0, i, S.w[i] * lam).index_add(0, k, -(1 - a) * wk * lam).index_add(0, k + 1, -a * wk1 * lam)
        return v

    S.hook = hook


def _four(a):
    return torch.cat([a, torch.zeros_like(a[..., :1])], -1)


def exact(case, seed):
    rods, drive, extra = _inputs(case, seed)
    S = _Rods64(rods)
    K, uhat = (a.double() for a in _joints(rods))
    if case["kind"] == "grad":
        return _grad64(S, case, K, uhat, torch.tensor(extra, device="cuda"))
    if case["kind"] == "vessel":
        _vessel64(S, rods[0], extra)
    elif case["kind"] == "knot":
        _knot64(S, rods[0], extra)
    elif case["kind"] == "pair":
        _pair64(S, case["n"], case["mode"])
    if drive is not None:
        drive = torch.tensor(drive, dtype=torch.float32, device="cuda").double()
    x, ticks = S.x, []
    for k in range(case.get("calls", 1)):
        d = None if drive is None else drive[k]
        if case["kind"] == "pair":
            S.beta = float(d[1, 3])
        for _ in range(case["steps"]):
            x = S.step(x, K, uhat, d)
        ticks.append(x[0])
    r, v, q, om = x
    out = {"quat": q, "vel": _four(v), "omega": _four(om)}
    if case["kind"] in ("rod", "vessel"):
        return {**out, "ticks": torch.stack(ticks), "inv_mass": S.w[:, 0].expand(len(ticks), -1)}
    return {**out, "pos": r, "inv_mass": S.w[:, 0]}


def _grad64(S, case, K, uhat, target):
    steps, every = case["steps"], case["every"]
    tips = torch.tensor(np.cumsum([case["n"]] * case["rods"]) - 1, device="cuda")
    marks, x = [], S.x
    traj = torch.empty((steps, S.E, 3), dtype=torch.float64, device="cuda")
    with torch.no_grad():
        for k in range(steps):
            if k % every == 0:
                marks.append(x)
            x = S.step(x, K, uhat, None)
            traj[k] = x[0]
    loss = (traj[:, tips] - target).square().sum()
    bar, kb, ub = [torch.zeros_like(a) for a in x], torch.zeros_like(K), torch.zeros_like(uhat)
    for m in reversed(range(len(marks))):  # a segment's steps again, then back through them
        leaves = [a.detach().clone().requires_grad_() for a in (*marks[m], K, uhat)]
        x, part = tuple(leaves[:4]), 0.0
        for k in range(m * every, min(steps, (m + 1) * every)):
            x = S.step(x, leaves[4], leaves[5], None)
            part = part + (x[0][tips] - target[k]).square().sum()
        part = part + sum((a * b).sum() for a, b in zip(x, bar))
        got = [torch.zeros_like(a) if g is None else g for a, g in zip(leaves, torch.autograd.grad(part, leaves, allow_unused=True))]
        bar, kb, ub = got[:4], kb + got[4], ub + got[5]
    return {"loss": loss, "traj": traj, "grad": {"K": kb, "uhat": ub, "vel": _four(bar[1]), "pos": _four(bar[0]),
                                                 "omega": _four(bar[3])}}
