"""The calls that users of this library make, as cases for timing and comparison.

A case is one whole run as a program makes it through the public entry points
(``Simulation``, ``Batch``, ``adjoint.rollout``): the initial condition from
an order-parameter field on the device, a number of time steps (with the fused
diagnostics where the case has them), and the fields read back; for the
adjoint, a rollout, a loss on the final field and its gradients.  Contexts,
batches with their tuned tiles, parameters and output arrays are made once in
``prepare``; a pass starts again from the initial field, so any number of
passes on one state gives the same outputs.

Fields come back in the precision that the run computes in: an FP32 run's
phi, p and u as float32.  ``exact`` is the same discrete model in plain
float64 torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_10827_gb300 import adjoint, sim, workloads

DEVICE = "cuda"

# Physical parameters of the runs, by the name used in a case.
PHYSICS = {
    # flat interfaces in FP64: the well-balance test
    "flat": workloads.physical(workloads.FLAT_16x128),
    # the stationary droplet of the throughput line (density ratio per case)
    "droplet": workloads.physical(workloads.DROPLET_1024),
    # the 128 x 128 droplet of the paper
    "droplet_paper": workloads.physical(workloads.DROPLET_PAPER),
    # two-droplet coalescence, 2D and 3D
    "coalescence": workloads.physical(workloads.COALESCENCE_ADJ),
    "coalescence3d": workloads.physical(workloads.COALESCENCE_3D),
}


def listed():
    return [
        # The smallest grid of the tests: flat interfaces, 16 x 128, FP64.  It
        # is run for 20 000 steps at a time, so the latency of a step counts.
        dict(name="slab_16x128_fp64", kind="run", nx=16, ny=128, nz=1, precision="fp64",
             physics="flat", init="slab", ratio=10.0, force=0.0, steps=400, diag=0),
        # The paper's droplet, 128 x 128: millions of steps to the steady
        # state in FP32, again bound by the latency of a step.
        dict(name="droplet_128_fp32", kind="run", nx=128, ny=128, nz=1, precision="fp32",
             physics="droplet_paper", init="droplet", ratio=10.0, force=0.0, steps=400, diag=0),
        # An ordinary run on a grid that divides into nothing: odd rows and
        # columns, a body force, diagnostics fused every 25 steps.
        dict(name="coalescence_301x203_fp32", kind="run", nx=301, ny=203, nz=1, precision="fp32",
             physics="coalescence", init="pair", ratio=10.0, force=1e-6, steps=200, diag=25),
        # The stationary droplet at the size of the throughput line, one grid
        # advanced by Simulation.step.
        dict(name="droplet_1024_fp32", kind="run", nx=1024, ny=1024, nz=1, precision="fp32",
             physics="droplet", init="droplet", ratio=10.0, force=0.0, steps=100, diag=0),
        # The throughput line: both density ratios in one batch, multi-step
        # launches, diagnostics every 20 steps.
        dict(name="pair_1024_batch_fp32", kind="batch", grids="pair", size=1024, count=2,
             precision="fp32", persistent=True, steps=60, diag=20),
        # The ensemble of 256 droplets on grids of 64 to 512 nodes a side.
        dict(name="ensemble_256_fp32", kind="batch", grids="ensemble", size=512, count=256,
             precision="fp32", persistent=False, steps=50, diag=0),
        # The FP64 run that FP32 results are checked against.
        dict(name="droplet_1024_fp64", kind="run", nx=1024, ny=1024, nz=1, precision="fp64",
             physics="droplet", init="droplet", ratio=100.0, force=0.0, steps=40, diag=0),
        # The small 3D coalescence used against the oracle.
        dict(name="coalescence3d_64_fp32", kind="run", nx=64, ny=64, nz=64, precision="fp32",
             physics="coalescence3d", init="pair", ratio=10.0, force=0.0, steps=100, diag=0),
        # The large 3D coalescence: 512^3, FP32.
        dict(name="coalescence3d_512_fp32", kind="run", nx=512, ny=512, nz=512, precision="fp32",
             physics="coalescence3d", init="pair", ratio=10.0, force=0.0, steps=20, diag=0),
        # 3D with FP16 offset storage, at a size that does not fit L2.
        dict(name="coalescence3d_256_f16off", kind="run", nx=256, ny=256, nz=256,
             precision="f16off", physics="coalescence3d", init="pair", ratio=10.0, force=0.0,
             steps=40, diag=0),
        # 3D with BF16 offset storage on a ragged grid, diagnostics (which
        # refresh the storage scales) every 20 steps.
        dict(name="coalescence3d_ragged_bf16off", kind="run", nx=100, ny=75, nz=130,
             precision="bf16off", physics="coalescence3d", init="pair", ratio=10.0, force=1e-6,
             steps=60, diag=20),
        # Gradients of a loss on the final field, 512 x 512 coalescence, FP32.
        dict(name="adjoint_512_fp32", kind="adjoint", nx=512, ny=512, precision="fp32",
             physics="coalescence", steps=400, every=100),
    ]


def draw(rng):
    """One more case of the same ranges (sizes over their logarithm)."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["2d", "2d", "2d64", "3d", "3d", "off", "off", "batch", "adjoint"])
    if what in ("2d", "2d64"):
        fp64 = what == "2d64"
        nx, ny = logint(24, 4096), logint(24, 4096 if not fp64 else 2048)
        return dict(kind="run", nx=nx, ny=ny, nz=1, precision="fp64" if fp64 else "fp32",
                    physics=_drawn_physics(rng, nx, ny),
                    init=rng.choice(["droplet", "pair", "slab"]),
                    ratio=round(rng.uniform(2.0, 100.0), 2),
                    force=rng.choice([0.0, 1e-6]),
                    steps=max(10, min(rng.randint(150, 450), int(1.0e8 / (nx * ny)))),
                    diag=rng.choice([0, 0, 20]))
    if what in ("3d", "off"):
        nx, ny, nz = logint(24, 320), logint(24, 320), logint(24, 320)
        return dict(kind="run", nx=nx, ny=ny, nz=nz,
                    precision=rng.choice(["f16off", "bf16off"]) if what == "off"
                    else rng.choice(["fp32", "fp32", "fp64"]),
                    physics="coalescence3d", init=rng.choice(["pair", "droplet"]),
                    ratio=round(rng.uniform(2.0, 50.0), 2), force=rng.choice([0.0, 1e-6]),
                    steps=max(10, min(rng.randint(60, 140), int(4.0e8 / (nx * ny * nz)))),
                    diag=rng.choice([0, 0, 20]))
    if what == "batch":
        grids = rng.choice(["pair", "ensemble"])
        return dict(kind="batch", grids=grids,
                    size=logint(64, 1400) if grids == "pair" else rng.randint(128, 512),
                    count=2 if grids == "pair" else logint(4, 128),
                    precision="fp32", persistent=rng.choice([True, False]),
                    steps=rng.randint(40, 100), diag=rng.choice([0, 20]))
    nx, ny = logint(32, 512), logint(32, 512)
    return dict(kind="adjoint", nx=nx, ny=ny, precision=rng.choice(["fp32", "fp32", "fp64"]),
                physics=_drawn_physics(rng, nx, ny), steps=rng.randint(50, 250),
                every=rng.choice([20, 50, 100]))


def _drawn_physics(rng, nx, ny):
    """Thick interfaces (W = 8) need some room."""
    return rng.choice(["droplet", "droplet_paper", "coalescence"] if min(nx, ny) >= 64
                      else ["droplet", "droplet_paper"])


# ------------------------------------------------------------------- inputs

def _offset(n, c):
    """Distance of the nodes 0 .. n-1 from c along a periodic axis."""
    x = torch.arange(n, dtype=torch.float64, device=DEVICE) - c
    return x - n * torch.round(x / n)


def _profile(d, W):
    return torch.tanh(2.0 * d / W)


def _blob(shape, centre, R, aspect, wave, W):
    """tanh profile of a deformed droplet: an ellipse(oid) with a surface wave."""
    dx, dy = _offset(shape[-1], centre[0]) / aspect, _offset(shape[-2], centre[1]) * aspect
    r2 = dx[None, :] ** 2 + dy[:, None] ** 2
    edge = R * (1.0 + wave * torch.cos(3.0 * torch.atan2(dy[:, None].expand_as(r2),
                                                         dx[None, :].expand_as(r2))))
    if len(shape) == 3:
        r2 = r2[None] + (_offset(shape[0], centre[2]) ** 2)[:, None, None]
    return _profile(edge - torch.sqrt(r2), W)


def _field(shape, init, W, rng, radius=None):
    """Initial order parameter of a grid (shape [nz,] ny, nx): droplets out of
    equilibrium (deformed, or about to merge) or a wavy slab."""
    nx, ny = shape[-1], shape[-2]
    c = [n * (0.5 + float(rng.uniform(-0.1, 0.1))) for n in (nx, ny) + tuple(shape[:-2])]
    if init == "slab":
        k = 2.0 * math.pi / nx
        x = torch.arange(nx, dtype=torch.float64, device=DEVICE)
        bump = float(rng.uniform(0.5, 1.5)) * torch.sin(k * x + float(rng.uniform(0.0, 6.28)))
        y = _offset(ny, c[1])
        return (0.5 + 0.5 * _profile(0.25 * ny + bump[None, :] - y.abs()[:, None],
                                     W)).contiguous()
    aspect, wave = float(rng.uniform(1.05, 1.2)), float(rng.uniform(0.02, 0.06))
    small = min(shape)
    if init == "droplet":
        R = (0.2 * small if radius is None else radius) * float(rng.uniform(0.9, 1.1))
        return (0.5 + 0.5 * _blob(shape, c, R, aspect, wave, W)).contiguous()
    # two droplets side by side, nearly touching (the coalescence formula)
    R = min(0.18 * nx, 0.25 * small) * float(rng.uniform(0.85, 1.0))
    half = R + 0.5 * W * float(rng.uniform(0.6, 1.0))
    a = _blob(shape, [c[0] - half] + c[1:], R, 1.0, wave, W)
    b = _blob(shape, [c[0] + half] + c[1:], R, 1.0, wave, W)
    return (0.5 + 0.5 * (1.0 + a + b)).contiguous()


def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case["nz"] > 1 else (case["ny"], case["nx"])


def _physics(case):
    p = dict(PHYSICS[case["physics"]])
    p["rho_l"] = case["ratio"] * p["rho_v"]
    if case["force"]:
        p["Gx"], p["Gy"] = case["force"], -0.5 * case["force"]
    return p


def _batch_grids(case, seed):
    """(n, radius, parameters, rng) of every grid of a batch."""
    out = []
    for c in range(case["count"]):
        p = dict(PHYSICS["droplet"])
        rng = np.random.default_rng([seed, c])
        if case["grids"] == "pair":
            n, R, ratio = case["size"], case["size"] / 8.0, (10.0, 100.0)[c % 2]
        else:
            # the ensemble recipe; the sizes are the case's, not the seed's
            e = workloads.ensemble_case(c)
            n = min(e["n"], case["size"])
            R, ratio = e["R"] * n / e["n"], e["rho_ratio"]
        p["rho_l"] = ratio * p["rho_v"]
        out.append((n, R, p, rng))
    return out


def _rng(seed):
    return np.random.default_rng([seed, 7])


def _diag_values(recs):
    """The records a monitoring program keeps: phi mass, energy, largest speed."""
    return {k: np.array([r[k] for r in recs], dtype=np.float32)
            for k in ("sum_phi", "kinetic_energy", "u_max")}


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "run":
        shape, prm = _shape(case), _physics(case)
        D = len(shape)
        s = sim.Simulation(shape[::-1], lattice="D2Q9" if D == 2 else "D3Q19",
                           precision=case["precision"], stream=stream, diag_every=case["diag"],
                           **prm)
        phi0 = _field(shape, case["init"], prm["W"], _rng(seed))
        out = {"phi": torch.empty(shape, dtype=torch.float64, device=DEVICE),
               "p": torch.empty(shape, dtype=torch.float64, device=DEVICE),
               "u": torch.empty((D,) + shape, dtype=torch.float64, device=DEVICE)}
        return dict(case=case, sim=s, phi0=phi0, out=out)
    if case["kind"] == "batch":
        grids = _batch_grids(case, seed)
        b = sim.Batch([((n, n), p) for n, _, p, _ in grids], precision=case["precision"],
                      stream=stream)
        phi0 = [_field((n, n), "droplet", p["W"], rng, R) for n, R, p, rng in grids]
        for i, f in enumerate(phi0):
            b.case(i).init_phi(f)
        # tiles are tuned once, as a program does before a long run
        if case["persistent"]:
            b.set_persistent(True)
        else:
            b.tune()
        b.set_diag_every(case["diag"])
        total = sum(f.numel() for f in phi0)
        out = {"phi": torch.empty(total, dtype=torch.float64, device=DEVICE),
               "p": torch.empty(total, dtype=torch.float64, device=DEVICE),
               "u": torch.empty(2 * total, dtype=torch.float64, device=DEVICE)}
        views, at = [], 0
        for f in phi0:
            n = f.numel()
            views.append((out["phi"][at:at + n], out["p"][at:at + n],
                          out["u"][2 * at:2 * (at + n)]))
            at += n
        return dict(case=case, batch=b, phi0=phi0, out=out, views=views)
    phi0, target, prm = _adjoint_inputs(case, seed)
    real = torch.float64 if case["precision"] == "fp64" else torch.float32
    leaf = lambda v: torch.tensor(v, dtype=real, device=DEVICE, requires_grad=True)  # noqa: E731
    return dict(case=case, phi0=phi0.to(real).requires_grad_(), target=target.to(real),
                sigma=leaf(prm.pop("sigma")), M=leaf(prm.pop("M")), prm=prm)


def _adjoint_inputs(case, seed):
    """Initial field, target field and parameters of an optimisation step: the
    target is another draw of the same two droplets."""
    prm = dict(PHYSICS[case["physics"]])
    shape = (case["ny"], case["nx"])
    phi0 = _field(shape, "pair", prm["W"], np.random.default_rng([seed, 8]))
    target = _field(shape, "pair", prm["W"], np.random.default_rng([seed, 9]))
    if case["precision"] != "fp64":
        phi0, target = phi0.float(), target.float()
    return phi0, target, prm


# --------------------------------------------------------------------- pass

def _as_computed(out, precision):
    return out if precision == "fp64" else {k: v.float() for k, v in out.items()}


def run(state):
    case = state["case"]
    if case["kind"] == "run":
        s, out = state["sim"], state["out"]
        s.init_phi(state["phi0"])
        s.step(case["steps"])
        s.moments_device(phi=out["phi"], p=out["p"], u=out["u"])
        got = dict(_as_computed(out, case["precision"]))
        if case["diag"]:
            got.update(_diag_values([s.last_diagnostics()]))
        return got
    if case["kind"] == "batch":
        b = state["batch"]
        for i, f in enumerate(state["phi0"]):
            b.case(i).init_phi(f)
        b.step(case["steps"])
        for i, (phi, p, u) in enumerate(state["views"]):
            b.case(i).moments_device(phi=phi, p=p, u=u)
        got = dict(_as_computed(state["out"], case["precision"]))
        if case["diag"]:
            got.update(_diag_values(b.last_diagnostics()))
        return got
    final = adjoint.rollout(state["phi0"].double(), state["sigma"], state["M"],
                            shape=(case["nx"], case["ny"]), nsteps=case["steps"],
                            checkpoint_every=case["every"], precision=case["precision"],
                            **state["prm"])
    final = final.to(state["target"].dtype)
    loss = ((final - state["target"]) ** 2).sum()
    g = torch.autograd.grad(loss, [state["phi0"], state["sigma"], state["M"]])
    return {"loss": loss.detach(), "final": final.detach(), "d_phi0": g[0], "d_sigma": g[1],
            "d_M": g[2]}


# --------------------------------------------------------------------- work

def work(case):
    """Bytes: every population and S read and written once per step in the
    storage format (f and g as Q values each; the offset formats also the six
    FP32 macroscopic fields), phi0 read and the fields written.  Operations:
    about 350 per D2Q9 and 800 per D3Q19 node update."""
    if case["kind"] == "adjoint":
        N, esz = case["nx"] * case["ny"], 8 if case["precision"] == "fp64" else 4
        # per node update: the recorded step (f, g, S read and written), its
        # recomputation (also writing five moments), and the reverse step
        # (f, g, moments, and the adjoints of f, phi, g, S read; the adjoints written)
        values = 38 + 38 + 5 + (18 + 5 + 20) + 20
        return dict(bytes=float(N * (case["steps"] * values * esz + 4 * esz)),
                    flops=float(N * case["steps"] * (2 * 350 + 1000)))
    if case["kind"] == "batch":
        N = sum(n * n for n, _, _, _ in _batch_grids(case, 0))
        D = 2
    else:
        N = case["nx"] * case["ny"] * case["nz"]
        D = 3 if case["nz"] > 1 else 2
    Q = 9 if D == 2 else 19
    per = {"fp32": 4 * Q * 4 + 8, "fp64": 4 * Q * 8 + 16, "f16off": 4 * Q * 2 + 2 * 24 + 8,
           "bf16off": 4 * Q * 2 + 2 * 24 + 8}[case["precision"]]
    field = 8 if case["precision"] == "fp64" else 4
    return dict(bytes=float(N * (case["steps"] * per + 8 + (2 + D) * field)),
                flops=float(N * case["steps"] * (350 if D == 2 else 800)))


# -------------------------------------------------------------------- exact

class _Model:
    """The discrete model in float64 torch operations.  ``at(v, c)`` is the
    field v taken at x + c: a roll of one periodic grid, or a gather over
    several grids laid end to end."""

    def __init__(self, D, at, W, sigma, M, alpha, rho_l, rho_v, nu_l, nu_v, force):
        if D == 2:
            cs = [(x, y) for y in (-1, 0, 1) for x in (-1, 0, 1)]
            weight = {0: 4.0 / 9.0, 1: 1.0 / 9.0, 2: 1.0 / 36.0}
            bias = {0: -2.0, 1: -0.5, 2: 1.0}
        else:
            cs = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)
                  if abs(x) + abs(y) + abs(z) < 3]
            weight = {0: 1.0 / 3.0, 1: 1.0 / 18.0, 2: 1.0 / 36.0}
            bias = {0: -2.5, 1: -1.0, 2: 0.5}
        self.D, self.at, self.force = D, at, force
        self.c = [c for c in cs if any(c)]
        self.w0, self.b0 = weight[0], bias[0]
        self.w = [weight[sum(map(abs, c))] for c in self.c]
        self.b = [bias[sum(map(abs, c))] for c in self.c]
        self.kappa, self.beta = 1.5 * W * sigma, 12.0 * sigma / W
        self.itf, self.alpha = 1.0 / (0.5 + 3.0 * M / alpha), alpha
        self.rho_v, self.drho = rho_v, rho_l - rho_v
        self.nu_v, self.dnu = nu_v, nu_l - nu_v

    def dot(self, c, v):
        s = None
        for k, ck in enumerate(c):
            if ck:
                s = ck * v[k] if s is None else s + ck * v[k]
        return s

    def mu(self, phi):
        lap = sum(w * (self.at(phi, c) - phi) for c, w in zip(self.c, self.w))
        return 4.0 * self.beta * phi * (phi - 1.0) * (phi - 0.5) - self.kappa * 6.0 * lap

    def grad(self, v):
        g = [0.0] * self.D
        for c, w in zip(self.c, self.w):
            s = self.at(v, c)
            g = [gk + 3.0 * w * ck * s if ck else gk for gk, ck in zip(g, c)]
        return g

    def start(self, phi):
        """(f_0, f_i, g_0, g_i, S_prev) of the initial condition, as arriving."""
        am = self.alpha * self.mu(phi)
        zero = torch.zeros_like(phi)
        return (phi - (1.0 - self.w0) * am, [w * am for w in self.w], zero,
                [zero] * len(self.c), zero)

    def moments(self, state):
        f0, f, g0, g, _ = state
        sf = sum(f)
        phi = f0 + sf
        mu = self.mu(phi)
        gp, gm = self.grad(phi), self.grad(mu)
        rho = self.rho_v + phi * self.drho
        F = [G - phi * gk for G, gk in zip(self.force, gm)]
        j = [0.5 * Fk for Fk in F]
        for c, gi in zip(self.c, g):
            j = [jk + ck * gi if ck else jk for jk, ck in zip(j, c)]
        u = [jk / rho for jk in j]
        gr = [self.drho * gk for gk in gp]
        uu = sum(uk * uk for uk in u)
        ugr = sum(uk * gk for uk, gk in zip(u, gr))
        p = (sum(g) + 0.5 * ugr - 1.5 * self.w0 * rho * uu) / (3.0 * (1.0 - self.w0))
        S = sum(uk * gk for uk, gk in zip(u, gp))
        return phi, mu, p, u, rho, F, gr, uu, S, sf

    def step(self, state):
        f0, f, g0, g, Sprev = state
        phi, mu, p, u, rho, F, gr, uu, S, sf = self.moments(state)
        am, Sh = self.alpha * mu, 1.5 * S - 0.5 * Sprev
        itg = 1.0 / (0.5 + 3.0 * (self.nu_v + phi * self.dnu))
        kg = 1.0 - 0.5 * itg
        n0 = f0 + self.itf * (sf - (1.0 - self.w0) * am) + self.w0 * self.b0 * Sh
        h0 = g0 + itg * (-3.0 * (1.0 - self.w0) * p - 1.5 * self.w0 * rho * uu - g0)
        base = 3.0 * p - 1.5 * rho * uu
        f, g = list(f), list(g)
        for i, (c, w, b) in enumerate(zip(self.c, self.w, self.b)):
            back = tuple(-k for k in c)
            f[i] = self.at(f[i] + self.itf * (w * am - f[i]) + w * b * Sh, back)
            cu, cF, cg = self.dot(c, u), self.dot(c, F), self.dot(c, gr)
            eq = w * (base + rho * cu * (3.0 + 4.5 * cu))
            g[i] = self.at(g[i] + itg * (eq - g[i]) + 3.0 * w * kg * (cF + cu * cg), back)
        return n0, f, h0, g, S

    def diagnostics(self, state):
        phi, _, _, _, rho, _, _, uu, _, _ = self.moments(state)
        return phi, 0.5 * rho * uu, uu


def _roll(v, c):
    return torch.roll(v, [-k for k in c[::-1]], dims=list(range(v.dim())))


def _model(prm, D, at, **other):
    q = dict(prm, **other)
    return _Model(D, at, q["W"], q["sigma"], q["M"], q["alpha"], q["rho_l"], q["rho_v"],
                  q["nu_l"], q["nu_v"], [q.get(k, 0.0) for k in ("Gx", "Gy", "Gz")[:D]])


def _last_diag(case):
    """Time of the last fused diagnostics of a run (they describe the state
    that a step starts from, at multiples of the cadence)."""
    return (case["steps"] - 1) // case["diag"] * case["diag"] if case["diag"] else -1


def _advance(model, state, case, split):
    """The state after the steps, and the diagnostics of each grid."""
    recs, last = None, _last_diag(case)
    for t in range(case["steps"]):
        if t == last:
            recs = [dict(sum_phi=float(phi.sum()), kinetic_energy=float(e.sum()),
                         u_max=math.sqrt(float(uu.max())))
                    for phi, e, uu in zip(*(split(v) for v in model.diagnostics(state)))]
        state = model.step(state)
    return state, recs


@torch.no_grad()
def _exact_run(case, seed):
    shape, prm = _shape(case), _physics(case)
    D = len(shape)
    model = _model(prm, D, _roll)
    state = model.start(_field(shape, case["init"], prm["W"], _rng(seed)))
    state, recs = _advance(model, state, case, lambda v: [v])
    m = model.moments(state)
    got = {"phi": m[0], "p": m[2], "u": torch.stack(m[3])}
    if recs:
        got.update({k: np.array([r[k] for r in recs]) for k in recs[0]})
    return got


@torch.no_grad()
def _exact_batch(case, seed):
    grids = _batch_grids(case, seed)
    phi0 = [_field((n, n), "droplet", p["W"], rng, R) for n, R, p, rng in grids]
    sizes = [f.numel() for f in phi0]
    index = {}
    for c in [(x, y) for y in (-1, 0, 1) for x in (-1, 0, 1)]:
        parts, at = [], 0
        for n, _, _, _ in grids:
            k = torch.arange(n, device=DEVICE)
            parts.append(at + (((k + c[1]) % n)[:, None] * n + ((k + c[0]) % n)[None, :]).ravel())
            at += n * n
        index[c] = torch.cat(parts)
    rho_l = torch.cat([torch.full((s,), p["rho_l"], dtype=torch.float64, device=DEVICE)
                       for s, (_, _, p, _) in zip(sizes, grids)])
    model = _model(PHYSICS["droplet"], 2, lambda v, c: v[index[c]], rho_l=rho_l)
    state = model.start(torch.cat([f.ravel() for f in phi0]))
    state, recs = _advance(model, state, case, lambda v: v.split(sizes))
    m = model.moments(state)
    u = torch.cat([torch.cat([a, b]) for a, b in zip(m[3][0].split(sizes), m[3][1].split(sizes))])
    got = {"phi": m[0], "p": m[2], "u": u}
    if recs:
        got.update({k: np.array([r[k] for r in recs]) for k in recs[0]})
    return got


def _exact_adjoint(case, seed):
    from torch.utils.checkpoint import checkpoint
    phi0, target, prm = _adjoint_inputs(case, seed)
    real = np.float64 if case["precision"] == "fp64" else np.float32
    leaf = lambda v: torch.tensor(float(real(v)), dtype=torch.float64, device=DEVICE,  # noqa: E731
                                  requires_grad=True)
    phi0 = phi0.double().requires_grad_()
    sigma, M = leaf(prm["sigma"]), leaf(prm["M"])
    Q = 8

    def segment(n, sigma, M, f0, g0, S, *fg):
        model = _model(prm, 2, _roll, sigma=sigma, M=M)
        state = (f0, list(fg[:Q]), g0, list(fg[Q:]), S)
        for _ in range(n):
            state = model.step(state)
        return (state[0], state[2], state[4], *state[1], *state[3])

    f0, f, g0, g, S = _model(prm, 2, _roll, sigma=sigma, M=M).start(phi0)
    flat = (f0, g0, S, *f, *g)
    left = case["steps"]
    while left > 0:
        n = min(20, left)
        flat = checkpoint(segment, n, sigma, M, *flat, use_reentrant=False)
        left -= n
    final = flat[0] + sum(flat[3:3 + Q])
    loss = ((final - target.double()) ** 2).sum()
    d = torch.autograd.grad(loss, [phi0, sigma, M])
    return {"loss": loss.detach(), "final": final.detach(), "d_phi0": d[0], "d_sigma": d[1],
            "d_M": d[2]}


def exact(case, seed):
    return {"run": _exact_run, "batch": _exact_batch, "adjoint": _exact_adjoint}[case["kind"]](
        case, seed)
