"""Performance cases of the lattice Boltzmann library: the calls that a
program built on it spends its time in, over the sizes, storage formats and
flows that the package's workloads, tests and benchmark use.

Every case builds a context on the GPU (``prepare``), runs one pass through
the public entry points (``run``) and can be evaluated in 64 bits by the plain
torch restatement at the end of this file (``exact``), which shares no code
with the package.

Kinds of pass:
  advance   n steps, then the canonical populations (and, in FP64, the wall
            force and the balance sums): stepping a flow towards its state
  drag      n steps, each with the drag on the body written to a device
            history, then the populations: the benchmark's loop
  monitor   the drag loop, then stress, balance and residual: what a run
            reports at an output interval
  exchange  a context filled from fields, exported, filled from exported
            populations (a restart file), exported again
  gradient  time-averaged drag and its gradient (forward and reverse run)
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2512_12213_gb300 import adjoint, lbm

BYTES = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the package's 2-D channel: 2,048 nodes, a step is a launch
        dict(name="channel_f64", kind="advance", flow="channel", nx=64, ny=32, nz=1, storage="f64", rounding="nearest",
             model="d", tau=0.8, steps=20),
        # Hartmann channel between a fixed and a moving wall: FP64 with the
        # Lorentz force, the configuration of the magnetohydrodynamic checks
        dict(name="hartmann_f64", kind="advance", flow="hartmann", nx=256, ny=128, nz=1, storage="f64",
             rounding="nearest", model="e", tau=0.8, steps=20),
        # flow past a sphere with the drag of every step: the benchmark
        dict(name="sphere_f16_drag", kind="drag", flow="sphere", nx=256, ny=128, nz=128, storage="f16s",
             rounding="stochastic", model="e", tau=0.68, steps=10),
        # the same flow in a box whose rows are no multiple of anything
        dict(name="sphere_ragged_bf16", kind="drag", flow="sphere", nx=250, ny=121, nz=99, storage="bf16s",
             rounding="stochastic", model="e", tau=0.536, steps=10),
        # FP32 run at an output interval: drag, stress tensors, balance, residual
        dict(name="sphere_f32_monitor", kind="monitor", flow="sphere", nx=256, ny=128, nz=128, storage="f32",
             rounding="nearest", model="e", tau=0.68, steps=10),
        # the FP64 reference run that the reduced formats are judged by
        dict(name="sphere_f64", kind="advance", flow="sphere", nx=128, ny=128, nz=128, storage="f64",
             rounding="nearest", model="e", tau=0.65, steps=5),
        # lid-driven cavity with the Smagorinsky model, FP32 and binary16
        dict(name="cavity_f32", kind="advance", flow="cavity", nx=256, ny=256, nz=256, storage="f32",
             rounding="nearest", model="e", tau=0.55, steps=10),
        dict(name="cavity_f16", kind="advance", flow="cavity", nx=256, ny=256, nz=256, storage="f16s",
             rounding="stochastic", model="e", tau=0.55, steps=10),
        # sphere in an imposed field with insulating walls (zero net current)
        dict(name="insulating_f32", kind="advance", flow="insulating", nx=256, ny=128, nz=128, storage="f32",
             rounding="nearest", model="e", tau=0.68, steps=10),
        # starting and restarting a large run
        dict(name="exchange_f16", kind="exchange", flow="cavity", nx=192, ny=192, nz=192, storage="f16s",
             rounding="nearest", model="e", tau=0.55, steps=0),
        # drag gradients of the 2-D cylinder and of a sphere
        dict(name="gradient_cylinder", kind="gradient", flow="cylinder", nx=512, ny=256, nz=1, storage="f32",
             rounding="nearest", model="e", tau=0.65, steps=40),
        dict(name="gradient_sphere", kind="gradient", flow="sphere", nx=128, ny=128, nz=128, storage="f32",
             rounding="nearest", model="e", tau=0.65, steps=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: 2-D flows of 32 x 16 to 1024 x 512 nodes, boxes of 40 x 24 x 24 to
    256 x 128 x 128 (cavities to 224^3), every storage format, force model and kind of pass."""
    kind = rng.choice(["advance", "advance", "drag", "drag", "monitor", "exchange", "gradient"])
    two_d = rng.random() < 0.35
    storage = rng.choice(["f64", "f32", "f32", "f16s", "f16s", "bf16s"])
    if kind == "gradient":
        flow, storage = ("cylinder" if two_d else "sphere"), rng.choice(["f32", "f32", "f64" if two_d else "f32", "f16s"])
    elif kind in ("drag", "monitor"):
        flow = "cylinder" if two_d else rng.choice(["sphere", "sphere", "brinkman", "curved"])
    else:
        flow = rng.choice(["channel", "hartmann", "cylinder"]) if two_d else rng.choice(
            ["sphere", "cavity", "cavity", "insulating", "brinkman", "curved"])
    if two_d:
        nx, ny, nz = _log(rng, 32, 1024), _log(rng, 16, 512), 1
    elif flow == "cavity":
        nx = ny = nz = _log(rng, 32, 128 if storage == "f64" else 224)
    else:
        side = 96 if storage == "f64" else 128
        nx, ny, nz = _log(rng, 40, 2 * side), _log(rng, 24, side), _log(rng, 24, side)
    if kind == "gradient":
        nx, ny = (min(nx, 512), min(ny, 256)) if two_d else (min(nx, 128), ny)
        steps = rng.randint(5, 40) if two_d else rng.randint(4, 12)
    elif kind == "exchange":
        steps = 0
    else:
        steps = rng.randint(4, 5) if storage == "f64" and not two_d else rng.randint(4, 10) if not two_d else \
            rng.randint(5, 40)
    rounding = rng.choice(["nearest", "stochastic"]) if storage in ("f16s", "bf16s") else "nearest"
    return dict(kind=kind, flow=flow, nx=nx, ny=ny, nz=nz, storage=storage, rounding=rounding,
                model=rng.choice(["a", "b", "c", "d", "e", "e", "e"]), tau=round(rng.uniform(0.55, 1.0), 3), steps=steps)


# ------------------------------------------------- configuration and geometry
def _config(case):
    """Keyword arguments of the context: the flows of the package's workloads at the case's size."""
    nx, ny, nz, tau, flow = case["nx"], case["ny"], case["nz"], case["tau"], case["flow"]
    cfg = dict(lattice=9 if nz == 1 else 19, nx=nx, ny=ny, nz=nz, periodic=(1, 1, 1), tau=tau, rho0=1.0,
               force_model=case["model"], g=(3.3e-7, 0.0, 0.0), storage=case["storage"], rounding=case["rounding"],
               seed=11, wall_u=((0.0, 0.0, 0.0),))
    if flow in ("channel", "hartmann"):
        cfg.update(periodic=(1, 0, 1), wall_u=((0.0, 0.0, 0.0), (0.0, 0.0, 0.0)), face_wall=(1, 1, 1, 2, 1, 1),
                   g=(1e-6, 0.0, 0.0))
    if flow == "hartmann":                 # Hartmann number 10, top wall moving
        K = (tau - 0.5) / 3 * 10.0 ** 2 / (ny / 2) ** 2
        cfg.update(g=(0.05 * K, 0.0, 0.0), lorentz=1, B=(0.0, 0.05, 0.0), sigma_e=K / 0.05 ** 2,
                   wall_u=((0.0, 0.0, 0.0), (0.05, 0.0, 0.0)))
    elif flow == "cylinder":
        cfg.update(g=(1.5e-6, 0.0, 0.0))
    elif flow == "insulating":
        cfg.update(lorentz=1, B=(0.0, 0.02, 0.0), sigma_e=1.0, insulating=1)
    elif flow == "brinkman":
        cfg.update(stokes=1, darcy=1e-4)
    elif flow == "curved":
        cfg.update(curved=1)
    elif flow == "cavity":                 # lid at +z moving along x
        cfg.update(periodic=(0, 0, 0), wall_u=((0.0, 0.0, 0.0), (0.1, 0.0, 0.0)), face_wall=(1, 1, 1, 1, 1, 2),
                   g=(0.0, 0.0, 0.0), les=1, cs=0.1)
    return cfg


def _geometry(case):
    """(solid mask uint8 (nz, ny, nx), signed distance to the body's surface or None)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    mask = np.zeros((nz, ny, nx), dtype=np.uint8)
    if case["flow"] in ("channel", "hartmann", "cavity"):
        return mask, None
    z, y, x = np.ogrid[0:nz, 0:ny, 0:nx]
    r2 = (x - nx // 4) ** 2 + (y - ny // 2) ** 2 + (0 if nz == 1 else (z - nz // 2) ** 2)
    radius = max(2, round(0.09 * min(ny, nz if nz > 1 else ny)))
    if case["flow"] == "curved":
        phi = (np.sqrt(r2) - (radius + 0.4)).astype(np.float32)
        mask[phi < 0] = 1
        return mask, phi
    mask[r2 <= radius * radius] = 1
    return mask, None


def _fields(case, seed):
    """Density and velocity of the start: a stream with a few smooth modes, float64 on the GPU."""
    g = np.random.default_rng(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    axes = [torch.arange(n, device="cuda", dtype=torch.float64) / n for n in shape]

    def smooth():
        s = torch.zeros(shape, device="cuda", dtype=torch.float64)
        for _ in range(3):
            k, ph = g.integers(0, 3, size=3), g.uniform(0, 2 * math.pi)
            s += torch.cos(2 * math.pi * (k[0] * axes[0][:, None, None] + k[1] * axes[1][None, :, None]
                                          + k[2] * axes[2][None, None, :]) + ph)
        return s / 3

    stream = 0.0 if case["flow"] == "cavity" else 0.05
    rho = 1.0 + 0.01 * smooth()
    u = 0.015 * torch.stack([smooth(), smooth(), smooth() if case["nz"] > 1 else torch.zeros_like(rho)])
    u[0] += stream
    return rho, u


def _populations(case, seed):
    """Canonical populations as a restart file holds them, on the GPU."""
    Q = 9 if case["nz"] == 1 else 19
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype, shape = _out_dtype(case), (case["nz"], case["ny"], case["nx"])
    f = torch.empty((Q,) + shape, dtype=dtype, device="cuda")
    for a in range(Q):
        f[a] = _WEIGHTS[Q][a] * (1.0 + 0.05 * (torch.rand(shape, generator=gen, device="cuda", dtype=dtype) - 0.5))
    return f


def _theta(seed):
    """Body force and wall velocity at which a gradient is taken."""
    g = np.random.default_rng(seed)
    return np.concatenate([g.uniform(0.5e-6, 2e-6, 1), g.uniform(-1e-7, 1e-7, 1), [0.0], g.uniform(-0.01, 0.01, 2), [0.0]])


def _out_dtype(case):
    return torch.float64 if case["storage"] == "f64" else torch.float32


# ------------------------------------------------------------ prepare and run
def prepare(case, seed):
    mask, phi = _geometry(case)
    sim = lbm.Sim(_config(case), mask, stage=case["kind"] == "gradient")    # the gradient starts from host arrays
    s = dict(case=case, sim=sim)
    if case["kind"] == "gradient":
        s["problem"] = adjoint.DragProblem(sim, case["steps"], 1)
        s["theta"] = torch.tensor(_theta(seed), dtype=torch.float32)
        return s
    if phi is not None:
        sim.set_wall_distance(phi)
    rho, u = _fields(case, seed)
    if case["kind"] == "exchange":
        s["rho"], s["u"] = rho, u
        s["f"] = _populations(case, seed)
        return s
    sim.init_equilibrium(rho, u)
    if case["kind"] != "advance":
        sim.step(2)                        # the wall force is that of a step taken
        s["history"] = torch.zeros((case["steps"], 3), dtype=torch.float64, device="cuda")
    if case["kind"] == "monitor":
        s["v_ref"] = sim.velocity_buffer()
    return s


def run(s):
    case, sim = s["case"], s["sim"]
    kind, dtype = case["kind"], _out_dtype(case)
    if kind == "gradient":
        theta = s["theta"].clone().requires_grad_(True)
        J = adjoint.DragFn.apply(theta, s["problem"])
        J.backward()
        return {"J": J.detach(), "gradient": theta.grad}
    if kind == "exchange":
        sim.init_equilibrium(s["rho"], s["u"])
        start = sim.export_f(dtype)
        sim.import_f(s["f"])
        return {"start": start, "restart": sim.export_f(dtype)}
    if kind == "advance":
        sim.step(case["steps"])
        out = {"f": sim.export_f(dtype)}
        if case["storage"] == "f64":
            mass, momentum, force = sim.balance()
            out.update(wall_force=sim.wall_force(), mass=mass, momentum=momentum, body_force=force)
        return out
    stream = sim.stream
    for i in range(case["steps"]):
        lbm.lbm_step_force(sim.ctx, 1, 0, 1.0, s["history"][i], lbm.OUT_DEVICE, stream)
    if kind == "drag":
        return {"force": s["history"], "f": sim.export_f(dtype)}
    sigma, strain, rho, v = sim.stress(lbm.S2)
    half, _, _, _ = sim.stress(lbm.S4)
    mass, momentum, force = sim.balance()
    change, total, _ = sim.residual(s["v_ref"])
    return {"force": s["history"], "sigma": sigma, "strain": strain, "rho": rho, "v": v, "sigma_half": half,
            "mass": mass, "momentum": momentum, "body_force": force, "change": change, "total": total}


def work(case):
    """Bytes and operations of one pass: per step every population read and
    written once; outputs and inputs in the type that the caller holds."""
    Q = 9 if case["nz"] == 1 else 19
    N, s = case["nx"] * case["ny"] * case["nz"], BYTES[case["storage"]]
    o = 8 if case["storage"] == "f64" else 4
    nc = 3 if Q == 9 else 6
    fl = 120 if Q == 9 else 270            # operations of a node update
    step, n, kind = 2 * Q * s, case["steps"], case["kind"]
    if kind == "gradient":
        # forward; one recomputed state and one reverse step per step but the last of each segment
        k = math.ceil(math.sqrt(n))
        again = n - math.ceil(n / k)
        return {"bytes": N * ((n + again) * step + n * Q * (s + 2 * o)), "flops": N * (2 * n + again) * fl}
    if kind == "exchange":
        return {"bytes": N * (4 * 8 + Q * o + 4 * Q * s + 2 * Q * o), "flops": N * 200}
    b = n * step
    if kind in ("advance", "drag"):
        b += Q * (s + o) + (Q * s if kind == "advance" and case["storage"] == "f64" else 0)
    else:
        b += 5 * Q * s + 2 * (2 * nc + 4) * o + 2 * 24
    return {"bytes": N * b, "flops": N * (n * fl + 100)}


# ----------------------------------------- the same passes in plain 64 bits
_WEIGHTS = {9: [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, 19: [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12}
_VELOCITIES = {
    9: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)],
    19: [(0, 0, 0)] + [tuple(s * c for c in e) for e in
                       [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
                       for s in (1, -1)],
}


class _Flow:
    """Collide and stream in float64 torch (dx = dt = 1).  Closed faces become
    a layer of solid nodes around the box, so that every axis can wrap."""

    def __init__(self, cfg, mask, phi=None):
        self.cfg, self.Q = cfg, cfg["lattice"]
        self.D = 2 if self.Q == 9 else 3
        new = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
        self.E, self.w = new(_VELOCITIES[self.Q]), new(_WEIGHTS[self.Q])
        self.vel = _VELOCITIES[self.Q]
        self.opp = [self.vel.index(tuple(-c for c in e)) for e in self.vel]
        m = mask.astype(np.int64)
        self.pad = [0 if cfg["periodic"][k] or (k == 2 and self.D == 2) else 1 for k in range(3)]   # x, y, z
        faces = cfg.get("face_wall", (1,) * 6)
        for k in (2, 1, 0):                # the first closed axis of x, y, z names a corner's wall
            if self.pad[k]:
                width = [(0, 0)] * 3
                width[2 - k] = (1, 1)
                m = np.pad(m, width, constant_values=((0, 0),) * (2 - k) + ((faces[2 * k], faces[2 * k + 1]),) +
                           ((0, 0),) * k)
        self.wall = torch.from_numpy(m).cuda()
        self.solid = self.wall > 0
        self.phi = None if phi is None else torch.from_numpy(phi.astype(np.float64)).cuda()
        self.g = new(cfg["g"])
        self.wall_u = torch.cat([torch.zeros(1, 3, dtype=torch.float64, device="cuda"), new(cfg["wall_u"])])
        self.B = new(cfg.get("B", (0.0, 0.0, 0.0)))
        self.field = torch.zeros(3, dtype=torch.float64, device="cuda")   # imposed electric field
        self.fluid = (~self.solid).double()

    def embed(self, t, fill=0.0):
        for k in (2, 1, 0):
            if self.pad[k]:
                t = torch.nn.functional.pad(t, [0] * (2 * k) + [1, 1], value=fill)
        return t

    def inner(self, t):
        for k in range(3):
            if self.pad[k]:
                t = t.narrow(t.dim() - 1 - k, 1, t.shape[t.dim() - 1 - k] - 2)
        return t

    def dot(self, x):
        return torch.tensordot(self.E, x, 1)

    def col(self, v):
        return v.view(-1, 1, 1, 1)

    def equilibrium(self, rho, u, linear=False):
        eu = self.dot(u)
        e = 1 + 3 * eu if linear else 1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0)
        return self.col(self.w) * rho * e

    def start(self, rho, u):
        return self.equilibrium(self.embed(rho, 1.0), self.embed(u), bool(self.cfg.get("stokes")))

    def macro(self, f):
        """rho, u^eq, u^F, v, A, C and tau of the node (force models a to e)."""
        c = self.cfg
        rho = f.sum(0)
        u = torch.tensordot(self.E.T, f, 1) / rho
        plane = self.col(torch.tensor([1.0, 1.0, 1.0 if self.D == 3 else 0.0], dtype=torch.float64, device="cuda"))
        A = self.col(self.g) * plane + 0 * u
        if c.get("lorentz") or c.get("darcy"):
            k, h, B = 0.5 * c.get("sigma_e", 0.0) / rho, 0.5 * c.get("darcy", 0.0), self.B
            Bp = self.col(B) * plane
            w = u + 0.5 * A + k * self.col(torch.linalg.cross(self.field, B)) * plane
            al, B2, Bp2 = 1 + h, (B * B).sum(), (Bp * Bp).sum()
            s = k * (Bp * w).sum(0) / (al + k * (B2 - Bp2))
            A = 2 * ((w + s * Bp) / (al + k * B2) - u)
        v = u + 0.5 * A
        model = c["force_model"]
        ueq = v if model == "e" else u
        tau = c["tau"]
        if c.get("les"):
            P = 0.0
            for i in range(self.D):
                for j in range(self.D):
                    p = torch.tensordot(self.E[:, i] * self.E[:, j], f, 1) - rho * ueq[i] * ueq[j]
                    P = P + (p - rho / 3 if i == j else p) ** 2
            tau = 0.5 * (tau + torch.sqrt(tau ** 2 + 18 * c["cs"] ** 2 * torch.sqrt(2 * P) / rho))
        C = 1 - 0.5 / tau if model == "e" else 1.0
        uF = {"a": 0 * u, "b": u, "c": u + 0.5 * tau * A, "d": v, "e": v}[model]
        return rho, ueq, uF, v, A, C, tau

    def collide(self, f):
        rho, ueq, uF, v, A, C, tau = self.macro(f)
        if self.cfg.get("insulating"):     # the next step's field: zero net current
            mean = (v * self.fluid).sum((1, 2, 3)) / self.fluid.sum()
            self.field = -torch.linalg.cross(mean, self.B)
        eA = self.dot(A)
        F = C * rho * self.col(self.w) * (3 * eA - 3 * (uF * A).sum(0) + 9 * self.dot(uF) * eA)
        return f + (self.equilibrium(rho, ueq, bool(self.cfg.get("stokes"))) - f) / tau + F

    def roll(self, t, e):
        return torch.roll(t, shifts=(e[2], e[1], e[0]), dims=(-3, -2, -1))

    def stream(self, P, u_w=None):
        """Pull with halfway (or interpolated) bounce-back and the moving-wall term."""
        u_w = self.wall_u if u_w is None else u_w
        out = []
        for b, e in enumerate(self.vel):
            if b == 0:
                out.append(P[0])
                continue
            a, hit = self.opp[b], self.roll(self.solid, e)
            L = 6 * self.w[b] * self.cfg["rho0"] * (u_w @ self.E[b])[self.roll(self.wall, e)]
            back = P[a] + L
            if self.phi is not None:
                q = self.phi / (self.phi - self.roll(self.phi, e))
                back_e = tuple(-c for c in e)
                near = 2 * q * P[a] + (1 - 2 * q) * self.roll(P[a], back_e) + L
                far = (P[a] + L) / (2 * q) + (1 - 1 / (2 * q)) * P[b]
                back = torch.where(q >= 0.5, far, torch.where(self.roll(self.solid, back_e), back, near))
            out.append(torch.where(hit, back, self.roll(P[b], e)))
        f = torch.stack(out)
        return torch.where(self.solid, self.col(self.w) * self.cfg["rho0"], f)

    def step(self, f):
        P = self.collide(f)
        return P, self.stream(P)

    def wall_force(self, P, f, wall=None):
        F = 0.0
        for b, e in enumerate(self.vel[1:], 1):
            a, at = self.opp[b], self.roll(self.wall, e)
            link = ((at > 0) if wall is None else (at == wall)) & ~self.solid
            F = F + self.E[a] * ((P[a] + f[b]) * link).sum()
        return F

    def canonical(self, f):
        return self.inner(torch.where(self.solid, torch.zeros_like(f), f))

    def balance(self, f):
        rho, _, _, _, A, _, _ = self.macro(f)
        m = torch.tensordot(self.E.T, f, 1)
        return ((rho * self.fluid).sum().item(), (m * self.fluid).sum((1, 2, 3)).cpu().numpy(),
                (rho * A * self.fluid).sum((1, 2, 3)).cpu().numpy())

    def pairs(self):
        return [(0, 0), (1, 1), (0, 1)] if self.D == 2 else [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]

    def stress(self, f):
        """Without the artefact term: sigma, strain rate, density, flow velocity."""
        rho, ueq, _, v, _, _, tau = self.macro(f)
        lin = bool(self.cfg.get("stokes"))
        sigma = torch.stack([-(1 - 0.5 / tau) * (torch.tensordot(self.E[:, i] * self.E[:, j], f, 1)
                                                 - (0 if lin else rho * ueq[i] * ueq[j]) - (rho / 3 if i == j else 0))
                             for i, j in self.pairs()])
        strain = sigma / (2 * rho * (tau - 0.5) / 3)
        return [self.canonical(t) for t in (sigma, strain, rho, v)]

    def stress_half(self, P, f, before):
        """At the half step, with the force's second moment: from f^rel(T-1), f(T) and f(T-1)."""
        fb = 0.5 * (P + f)
        rb = fb.sum(0)
        ub = torch.tensordot(self.E.T, fb, 1) / rb
        rho, _, uF, _, A, C, _ = self.macro(before)
        lin, on = bool(self.cfg.get("stokes")), self.cfg["force_model"] != "a"
        return self.canonical(torch.stack([
            -(torch.tensordot(self.E[:, i] * self.E[:, j], fb, 1) - (0 if lin else rb * ub[i] * ub[j])
              - (rb / 3 if i == j else 0)) + (0.5 * C * rho * (uF[i] * A[j] + uF[j] * A[i]) if on else 0)
            for i, j in self.pairs()]))


def _exact_gradient(case, flow, seed):
    theta = torch.tensor(_theta(seed), dtype=torch.float32).double().cuda().requires_grad_(True)
    shape = (case["nz"], case["ny"], case["nx"])
    rest = torch.ones(shape, dtype=torch.float64, device="cuda")
    f = flow.start(rest, torch.zeros((3,) + shape, dtype=torch.float64, device="cuda"))
    T = case["steps"]

    def one(f, theta):
        flow.g = theta[:3]
        u_w = torch.cat([torch.zeros(1, 3, dtype=torch.float64, device="cuda"), theta[3:].view(1, 3)])
        P = flow.collide(f)
        g = flow.stream(P, u_w)
        return g, flow.wall_force(P, g, 1)[0] / T

    J = 0.0
    for _ in range(T):
        f, F = torch.utils.checkpoint.checkpoint(one, f, theta, use_reentrant=False)
        J = J + F
    J.backward()
    return {"J": J.detach().cpu(), "gradient": theta.grad.detach().cpu()}


def exact(case, seed):
    cfg = _config(case)
    mask, phi = _geometry(case)
    flow = _Flow(cfg, mask, phi)
    if case["kind"] == "gradient":
        return _exact_gradient(case, flow, seed)
    rho, u = _fields(case, seed)
    with torch.no_grad():
        f = flow.start(rho, u)
        if case["kind"] == "exchange":
            given = _populations(case, seed).double()
            return {"start": flow.canonical(f), "restart": given * (~flow.inner(flow.solid))}
        history = []
        for i in range(case["steps"] + (0 if case["kind"] == "advance" else 2)):
            before = f
            if case["kind"] != "advance" and i >= 2:
                history.append(flow.wall_force(P, f, 1))
            P, f = flow.step(f)
        out = {"f": flow.canonical(f)}
        if case["kind"] == "advance":
            if case["storage"] == "f64":
                mass, momentum, force = flow.balance(f)
                out.update(wall_force=flow.wall_force(P, f).cpu().numpy(), mass=mass, momentum=momentum,
                           body_force=force)
            return out
        out["force"] = torch.stack(history)
        if case["kind"] == "drag":
            return out
        sigma, strain, rho, v = flow.stress(f)
        mass, momentum, force = flow.balance(f)
        total = (v.square().sum(0).sqrt()).sum().item()
        return {"force": out["force"], "sigma": sigma, "strain": strain, "rho": rho, "v": v,
                "sigma_half": flow.stress_half(P, f, before), "mass": mass, "momentum": momentum, "body_force": force,
                "change": total, "total": total}
