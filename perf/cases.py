"""Workloads of the framework, as a user's program runs them.

Each case is one pass of something that the programs of this repository do over and
over through its public entry points: time steps of one run, of a batch of runs and of
a 3-D run, the measurements taken between steps, and the surrogate network's fit and
scan.  Sizes are those of the benchmark, the Table 1 and sweep programs, the metrics log
and the tests; drawn cases spread over the same ranges.

Kinds of case:
  step    Sim.step(steps), then the macroscopic fields into device arrays
  label   a new run: fields in, steps, diagnostics and drop count (what a sweep does per run)
  batch   Batch.step(steps) of many runs, then every run's fields
  step3   the 3-D lattices: steps, then phi and c
  fit     Surrogate.train on labelled points, then the parameters
  scan    Surrogate.predict over a dense scan of points
Snapshots of fields are kept in single precision, the precision the steps compute in.
"""
import math

import numpy as np
import torch

from paper_2504_09024_gb300 import lbm, lbm3, workloads

DTYPES = {"f32": lbm.LBM_F32, "f16": lbm.LBM_F16S, "bf16": lbm.LBM_BF16S}
WORDS = {"f32": 4, "f16": 2, "bf16": 2}
SCAN_CAS = 46  # capillary numbers 0.05, 0.06, ..., 0.5 of a scan

_stream = None


def stream():
    """The one CUDA stream such a program runs everything on."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def _step(nx, ny, steps, dtype="f32", walls=1, fixed_u=False, ratio=1.0, tune=False, kind="step"):
    return {"kind": kind, "nx": nx, "ny": ny, "steps": steps, "dtype": dtype, "walls": walls,
            "fixed_u": fixed_u, "ratio": ratio, "tune": tune}


def listed():
    return [
        # the benchmark's drop in shear, launch shape from the autotuner as the benchmark does
        dict(name="shear-2048x1024-f32", **_step(2048, 1024, 64, tune=True)),
        # the same grid in 16-bit storage with the library's own launch shape
        dict(name="shear-2048x1024-f16", **_step(2048, 1024, 64, dtype="f16")),
        # the metrics log's drop, stepped between two records
        dict(name="shear-512x256-f32", **_step(512, 256, 64)),
        # the surfactant on a drop at rest under a prescribed velocity: the smallest calls
        dict(name="fixed-u-128x128-f32", **_step(128, 128, 50, walls=0, fixed_u=True)),
        # a ragged periodic grid with density and viscosity ratios and BF16 storage
        dict(name="ratio-301x167-bf16", **_step(301, 167, 40, dtype="bf16", walls=0, ratio=2.0)),
        # one labelled run: new fields, steps, deformation, drop count
        dict(name="label-1024x512-f32", **_step(1024, 512, 16, kind="label")),
        # Table 1: ten runs of 768 x 256 as one batch
        {"name": "table1-10x768x256", "kind": "batch", "nx": 768, "ny": 256, "runs": 10, "steps": 32},
        # the sweep's held-out points: 128 runs of 384 x 128 as one batch
        {"name": "sweep-128x384x128", "kind": "batch", "nx": 384, "ny": 128, "runs": 128, "steps": 16},
        # the 3-D benchmark: a spherical drop advected by a uniform velocity
        {"name": "sphere-256", "kind": "step3", "nx": 256, "ny": 256, "nz": 256, "steps": 8, "field": False},
        # a smaller ragged box in a velocity field
        {"name": "sphere-field-150x97x61", "kind": "step3", "nx": 150, "ny": 97, "nz": 61, "steps": 16,
         "field": True},
        # fitting the surrogate to a sweep's 1024 labelled runs (64 of its 3000 epochs)
        {"name": "fit-1024", "kind": "fit", "n": 1024, "epochs": 64},
        # scanning 256 sweep points for their critical capillary number
        {"name": "scan-256", "kind": "scan", "n": 256 * SCAN_CAS},
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "label", "batch", "step3", "step3", "fit", "scan"])
    if kind in ("step", "label"):
        ny = _spread(rng, 64, 1024)
        nx = min(2048, max(64, int(ny * rng.uniform(0.9, 3.1))))
        walls = rng.choice([0, 1, 1])
        fixed = kind == "step" and rng.random() < 0.3
        dtype = rng.choice(["f32", "f32", "f16", "bf16"])
        ratio = 1.0 if fixed or rng.random() < 0.6 else round(rng.uniform(1.1, 3.0), 3)
        steps = _spread(rng, 8, 64) if kind == "step" else _spread(rng, 8, 32)
        return _step(nx, ny, steps, dtype=dtype, walls=0 if fixed else walls, fixed_u=fixed,
                     ratio=ratio, kind=kind)
    if kind == "batch":
        ny = _spread(rng, 64, 256)
        nx = int(ny * rng.uniform(1.5, 3.1))
        runs = _spread(rng, 2, max(3, min(128, 6300000 // (nx * ny))))
        return {"kind": "batch", "nx": nx, "ny": ny, "runs": runs, "steps": _spread(rng, 8, 32)}
    if kind == "step3":
        n = _spread(rng, 24, 220)
        a, b = rng.uniform(0.6, 1.1), rng.uniform(0.4, 1.1)
        return {"kind": "step3", "nx": n, "ny": max(16, int(a * n)), "nz": max(16, int(b * n)),
                "steps": _spread(rng, 4, 16 if n < 160 else 8), "field": rng.random() < 0.5}
    if kind == "fit":
        return {"kind": "fit", "n": _spread(rng, 64, 1500), "epochs": _spread(rng, 8, 64)}
    return {"kind": "scan", "n": SCAN_CAS * _spread(rng, 8, 256) - rng.randrange(SCAN_CAS)}


def work(case):
    kind = case["kind"]
    if kind in ("step", "label", "batch"):
        cells = case["nx"] * case["ny"] * case.get("runs", 1)
        lattices = 2 if case.get("fixed_u") else 3
        pop = 2 * 9 * lattices * WORDS[case.get("dtype", "f32")]  # populations read and written
        out = 4 * 5 if kind != "label" else 8 * 4                 # fields out, or fields in
        flops = 300 if case.get("fixed_u") else 600
        return {"bytes": cells * (pop * case["steps"] + out), "flops": cells * flops * case["steps"]}
    if kind == "step3":
        cells = case["nx"] * case["ny"] * case["nz"]
        per = 2 * 27 * 2 * 4 + (12 if case["field"] else 0)
        return {"bytes": cells * (per * case["steps"] + 8), "flops": cells * 700 * case["steps"]}
    weights = 5 * 128 + 3 * 128 * 128 + 128 * 2
    n = case["n"]
    if kind == "fit":
        state = 4 * 4 * weights  # parameters, their gradients and both Adam moments
        return {"bytes": case["epochs"] * 2 * state + 28 * n, "flops": 6 * n * weights * case["epochs"]}
    return {"bytes": 28 * n + 4 * weights, "flops": 2 * n * weights}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _grid(nx, ny):
    x = torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5
    y = torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5
    return x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)


def _run_2d(nx, ny, rng, walls, fixed_u=False, ratio=1.0):
    """Physics and fields of one run: a drop in shear between moving walls (walls), a
    drop in a periodic box with a uniform stream, or the surfactant on a drop under a
    prescribed velocity (fixed_u)."""
    W = 4.0 if ny < 1024 else 5.0
    R = min(nx, ny) * rng.uniform(0.17, 0.22)
    xc = nx * 0.5 + rng.uniform(-0.05, 0.05) * nx
    yc = ny * 0.5 + rng.uniform(-0.03, 0.03) * ny
    gamma0 = rng.uniform(0.1, 0.45)
    if fixed_u:
        U = rng.uniform(0.0, 0.01)
        phys = workloads.Physics(nx=nx, ny=ny, walls_y=0, mode=1, W=W, M_phi=0.1, D_s=rng.uniform(0.05, 0.2))
    elif walls:
        d = workloads.shear_drop_parameters(ny, R, W, 0.1, 1.0, Re=rng.uniform(0.1, 1.0),
                                            Ca=rng.uniform(0.05, 0.5),
                                            Pe_s=math.exp(rng.uniform(0.0, math.log(10.0))))
        U = d.U_o
        phys = workloads.Physics(nx=nx, ny=ny, walls_y=1, mode=0, u_wall=U, W=W, M_phi=d.M_phi, D_s=d.D_s,
                                 nu_a=0.1 * ratio, nu_b=0.1, rho_a=ratio, rho_b=1.0, sigma_o=d.sigma_o,
                                 beta=rng.uniform(0.0, 0.5), c_max=1.0)
    else:
        U = rng.uniform(0.005, 0.02)
        phys = workloads.Physics(nx=nx, ny=ny, walls_y=0, mode=0, W=W, M_phi=0.02, D_s=0.02,
                                 nu_a=0.1 * ratio, nu_b=0.1, rho_a=ratio, rho_b=1.0, sigma_o=5e-3, beta=0.3,
                                 c_max=1.0)
    X, Y = _grid(nx, ny)
    dx, dy = X - xc, Y - yc
    # sheared drops are stretched along the diagonal
    a = 1.0 if fixed_u else rng.uniform(1.05, 1.25)
    along, across = (dx + dy) / math.sqrt(2.0) / a, (dy - dx) / math.sqrt(2.0) * a
    zeta = R - torch.hypot(along, across)
    phi = 0.5 + 0.5 * torch.tanh(2.0 * zeta / W)
    c = (gamma0 + 0.1 * torch.cos(torch.atan2(dy, dx))) / torch.cosh((2.0 * zeta / W).clamp(-300.0, 300.0)) ** 2
    ux = U * (2.0 * Y / ny - 1.0) if walls and not fixed_u else torch.full_like(phi, U)
    return phys, tuple(v.contiguous() for v in (phi, c, ux, torch.zeros_like(phi)))


def _inputs_2d(case, seed):
    rng = np.random.default_rng([2504, seed])
    return _run_2d(case["nx"], case["ny"], rng, case["walls"], case["fixed_u"], case["ratio"])


def _inputs_batch(case, seed):
    rng = np.random.default_rng([9024, seed])
    return [_run_2d(case["nx"], case["ny"], rng, 1) for _ in range(case["runs"])]


def _inputs_3d(case, seed):
    rng = np.random.default_rng([27, seed])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    z = (torch.arange(nz, dtype=torch.float64, device="cuda") + 0.5)[:, None, None]
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5)[None, :, None]
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5)[None, None, :]
    R, W = 0.25 * min(nx, ny, nz), 4.0
    at = [n * (0.5 + rng.uniform(-0.05, 0.05)) for n in (nx, ny, nz)]
    dx, dy, dz = x - at[0], y - at[1], z - at[2]
    r = torch.sqrt(dx * dx + dy * dy + dz * dz)
    phi = 0.5 + 0.5 * torch.tanh(2.0 * (R - r) / W)
    mode = rng.uniform(0.05, 0.15) * dz / r.clamp_min(1e-6)
    c = (0.5 + mode) / torch.cosh((2.0 * (R - r) / W).clamp(-300.0, 300.0)) ** 2
    if case["field"]:
        # a divergence-free vortex with a mean drift
        a, k = rng.uniform(0.01, 0.04), 2.0 * math.pi
        one = torch.ones_like(phi)
        u = (a * torch.sin(k * x / nx) * torch.cos(k * y / ny) * one,
             -a * ny / nx * torch.cos(k * x / nx) * torch.sin(k * y / ny) * one, 0.01 * one)
        u = tuple(v.contiguous() for v in u)
    else:
        u = tuple(float(v) for v in rng.uniform(-0.025, 0.025, 3))
    return phi.contiguous(), c.contiguous(), u, W


def _inputs_net(case, seed):
    rng = np.random.default_rng([5, seed])
    n = case["n"]
    if case["kind"] == "scan":
        points = np.repeat(rng.uniform(-1.0, 1.0, (-(-n // SCAN_CAS), 5)), SCAN_CAS, axis=0)
        points[:, 0] = np.tile(np.linspace(-1.0, 1.0, SCAN_CAS), len(points) // SCAN_CAS)
        return points[:n].astype(np.float32)
    X = rng.uniform(-1.0, 1.0, (n, 5)).astype(np.float32)
    stretch = 0.22 + 0.16 * X[:, 0] + 0.05 * X[:, 1] * X[:, 3] + 0.03 * X[:, 4]
    return X, stretch.astype(np.float32), (stretch > 0.27).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("fit", "scan"):
        return {"case": case, "net": lbm.Surrogate(seed=seed % 1000003), "data": _inputs_net(case, seed)}
    s = stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        if kind == "step3":
            phi, c, u, W = _inputs_3d(case, seed)
            sim = lbm3.Sim3(case["nx"], case["ny"], case["nz"], W=W, M_phi=0.05, D_s=0.1,
                            u=(0.0, 0.0, 0.0) if case["field"] else u, velocity_field=case["field"],
                            stream=s.cuda_stream)
            lbm3.lbm3_init_fields_device(sim.ctx, phi, c, *(u if case["field"] else (None, None, None)))
            out = torch.empty((2,) + sim.shape, dtype=torch.float64, device="cuda")
            return {"case": case, "sim": sim, "out": out, "keep": (phi, c, u)}
        if kind == "batch":
            runs = _inputs_batch(case, seed)
            batch = lbm.Batch([p for p, _ in runs], stream=s.cuda_stream)
            for r, (_, fields) in zip(batch.runs, runs):
                lbm.lbm_init_fields_device(r.ctx, *fields)
            out = torch.empty((case["runs"], 5, case["ny"], case["nx"]), dtype=torch.float64, device="cuda")
            return {"case": case, "batch": batch, "out": out, "keep": runs}
        phys, fields = _inputs_2d(case, seed)
        sim = lbm.Sim(phys, dtype=DTYPES[case["dtype"]], stream=s.cuda_stream)
        if kind == "step":
            lbm.lbm_init_fields_device(sim.ctx, *fields)
            if case["tune"]:
                sim.autotune(steps=32)
        out = torch.empty((5, case["ny"], case["nx"]), dtype=torch.float64, device="cuda")
        return {"case": case, "sim": sim, "out": out, "fields": fields}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _snapshot(sim, out):
    """The macroscopic fields of a run, into the program's device arrays."""
    lbm.lbm_get_fields_device(sim.ctx, out[0], out[1], out[2], out[3], out[4])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "fit":
        X, yD, yB = state["data"]
        loss = state["net"].train(X, yD, yB, epochs=case["epochs"], lr=2e-3)
        return {"loss": loss, "params": state["net"].get_params()}
    if kind == "scan":
        D, logit = state["net"].predict(state["data"])
        return {"D": D, "logit": logit}
    out = state["out"]
    with torch.cuda.stream(stream()):
        if kind == "step3":
            state["sim"].step(case["steps"])
            lbm3.lbm3_get_fields_device(state["sim"].ctx, out[0], out[1])
            kept = out.float()
            return {"phi": kept[0], "c": kept[1]}
        if kind == "batch":
            batch = state["batch"]
            batch.step(case["steps"])
            for k, r in enumerate(batch.runs):
                _snapshot(r, out[k])
            kept = out.float()
            return {"phi": kept[:, 0], "c": kept[:, 1], "u": kept[:, 2:4], "P": kept[:, 4]}
        sim = state["sim"]
        if kind == "label":
            lbm.lbm_init_fields_device(sim.ctx, *state["fields"])
            sim.step(case["steps"])
            found = sim.diagnostics()
            found["drops"] = sim.components(0.5)
            return found
        sim.step(case["steps"])
        _snapshot(sim, out)
        kept = out.float()
        return {"phi": kept[0], "c": kept[1], "u": kept[2:4], "P": kept[4]}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

CS2 = 1.0 / 3.0
E1 = (0, 1, -1)             # one-dimensional velocities, in the order used below
W1 = (2.0 / 3.0, 1.0 / 6.0, 1.0 / 6.0)


def _to_central(a, u):
    """Central moments of order 0, 1, 2 along one axis of the three populations a."""
    return [a[0] + a[1] + a[2],
            -u * a[0] + (1.0 - u) * a[1] - (1.0 + u) * a[2],
            u * u * a[0] + (1.0 - u) ** 2 * a[1] + (1.0 + u) ** 2 * a[2]]


def _from_central(k, u):
    """The populations along one axis that have the central moments k."""
    u2 = u * u
    return [(1.0 - u2) * k[0] - 2.0 * u * k[1] - k[2],
            0.5 * (u2 + u) * k[0] + (u + 0.5) * k[1] + 0.5 * k[2],
            0.5 * (u2 - u) * k[0] + (u - 0.5) * k[1] + 0.5 * k[2]]


def _central2(a, ux, uy):
    rows = [_to_central([a[0][n], a[1][n], a[2][n]], ux) for n in range(3)]  # rows[n][m]
    return [_to_central([rows[0][m], rows[1][m], rows[2][m]], uy) for m in range(3)]


def _populations2(k, ux, uy):
    cols = [_from_central([k[0][n], k[1][n], k[2][n]], ux) for n in range(3)]
    return [_from_central([cols[0][a], cols[1][a], cols[2][a]], uy) for a in range(3)]


class _Exact2:
    """The coupled D2Q9 step; a lattice is a[ix][iy] with velocities E1[ix], E1[iy]."""

    def __init__(self, phys, fields):
        self.p = p = phys
        self.dphi = p.phi_a - p.phi_b
        phi, c, ux, uy = fields
        self.u = (ux, uy)
        zero = torch.zeros_like(phi)
        gx, gy = self.gradient(phi)
        nx, ny, _ = self.normal(gx, gy)
        theta, theta_c = self.interface(phi, c)
        self.f = _populations2(self.scalar(phi, p.M_phi * theta * nx, p.M_phi * theta * ny, zero), ux, uy)
        self.h = _populations2(self.scalar(c, p.D_s * theta_c * nx, p.D_s * theta_c * ny, zero), ux, uy)
        if p.mode == 0:
            P = torch.full_like(phi, 0.5 * CS2 * (p.rho_a + p.rho_b))
            self.g = _populations2(self.flow_equilibrium(self.between(phi, p.rho_a, p.rho_b), P, ux, uy), ux, uy)

    def shifted(self, v, dx, dy, odd=False):
        """v at x + (dx, dy); rows beyond a wall mirror those inside (odd: with the sign changed)."""
        v = torch.roll(v, -dx, 1) if dx else v
        if not dy:
            return v
        w = torch.roll(v, -dy, 0)
        if self.p.walls_y:
            edge = -1 if dy > 0 else 0
            w[edge] = -v[edge] if odd else v[edge]
        return w

    def gradient(self, v, odd=False):
        at = {(a, b): self.shifted(v, a, b, odd) for a in (-1, 0, 1) for b in (-1, 0, 1) if a or b}
        gx = (at[1, 0] - at[-1, 0]) / 3.0 + (at[1, 1] - at[-1, 1] + at[1, -1] - at[-1, -1]) / 12.0
        gy = (at[0, 1] - at[0, -1]) / 3.0 + (at[1, 1] - at[1, -1] + at[-1, 1] - at[-1, -1]) / 12.0
        return gx, gy

    @staticmethod
    def normal(gx, gy):
        m = torch.sqrt(gx * gx + gy * gy)
        inv = torch.where(m > 1e-12, 1.0 / m, torch.zeros_like(m))
        return gx * inv, gy * inv, m

    def between(self, phi, a, b):
        return b + (phi - self.p.phi_b) / self.dphi * (a - b)

    def interface(self, phi, c):
        p = self.p
        theta = 4.0 / p.W * (p.phi_a - phi) * (phi - p.phi_b) / self.dphi
        return theta, 8.0 * c / p.W * (0.5 * (p.phi_a + p.phi_b) - phi) / self.dphi

    @staticmethod
    def scalar(s, kx, ky, zero):
        return [[s, ky, CS2 * s], [kx, zero, zero], [CS2 * s, zero, CS2 * CS2 * s]]

    @staticmethod
    def flow_equilibrium(rho, P, ux, uy):
        R = rho * CS2
        M = (1.0, 0.0, CS2)
        Wx, Wy = (1.0, -ux, ux * ux + CS2), (1.0, -uy, uy * uy + CS2)
        return [[R * (M[m] * M[n]) + (P - R) * (Wx[m] * Wy[n]) for n in range(3)] for m in range(3)]

    def macroscopic(self):
        p = self.p
        total = lambda a: sum(v for col in a for v in col)  # noqa: E731
        phi, c = total(self.f), total(self.h)
        nx, ny, m = self.normal(*self.gradient(phi))
        d = {"phi": phi, "c": c, "nx": nx, "ny": ny}
        if p.mode != 0:
            d.update(ux=self.u[0], uy=self.u[1], P=torch.zeros_like(phi))
            return d
        Ps = total(self.g)
        kappa = self.gradient(nx)[0] + self.gradient(ny, odd=True)[1]
        sigma = p.sigma_o * (1.0 + p.beta * torch.log(1.0 - c / p.c_max)) if p.beta else torch.full_like(c, p.sigma_o)
        sx, sy = self.gradient(sigma)
        along = nx * sx + ny * sy
        N = 1.5 * p.W / self.dphi ** 2 * m * m
        Ftx = N * (sx - nx * along - sigma * kappa * nx) + p.fext_x
        Fty = N * (sy - ny * along - sigma * kappa * ny) + p.fext_y
        rho = self.between(phi, p.rho_a, p.rho_b)
        jx, jy = sum(self.g[1]) - sum(self.g[2]), sum(v[1] for v in self.g) - sum(v[2] for v in self.g)
        ux, uy = (jx + 0.5 * CS2 * Ftx) / (CS2 * rho), (jy + 0.5 * CS2 * Fty) / (CS2 * rho)
        px, py = self.gradient(Ps - CS2 * rho)
        G = -px * ux - py * uy
        d.update(ux=ux, uy=uy, P=Ps + 0.5 * G, Ft=(Ftx, Fty), Fp=(-px, -py), rho=rho, G=G)
        return d

    def step(self):
        p, d = self.p, self.macroscopic()
        phi, c, ux, uy = d["phi"], d["c"], d["ux"], d["uy"]
        zero = torch.zeros_like(phi)
        theta, theta_c = self.interface(phi, c)

        def relaxed(a, s, K, t):
            w = 1.0 / (3.0 * K + 0.5)
            jx, jy = sum(a[1]) - sum(a[2]), sum(v[1] for v in a) - sum(v[2] for v in a)
            kx, ky = jx - ux * s, jy - uy * s
            k = self.scalar(s, kx + w * (K * t * d["nx"] - kx), ky + w * (K * t * d["ny"] - ky), zero)
            return self.streamed(_populations2(k, ux, uy))

        self.f = relaxed(self.f, phi, p.M_phi, theta)
        self.h = relaxed(self.h, c, p.D_s, theta_c)
        if p.mode != 0:
            return
        rho, G, (Fx, Fy), (Tx, Ty) = d["rho"], d["G"], d["Fp"], d["Ft"]
        eq = self.flow_equilibrium(rho, d["P"], ux, uy)
        k = _central2(self.g, ux, uy)
        w_nu = 1.0 / (3.0 * self.between(phi, p.nu_a, p.nu_b) + 0.5)
        w_zeta = 1.0 / (3.0 * p.zeta + 0.5)
        s20 = 2.0 * CS2 * Fx * ux + (ux * ux + CS2) * G
        s02 = 2.0 * CS2 * Fy * uy + (uy * uy + CS2) * G
        s11 = CS2 * (Fx * uy + Fy * ux) + ux * uy * G

        def mixed(now, goal, source, w):
            return now + w * (goal - now) + (1.0 - 0.5 * w) * source

        both = mixed(k[2][0] + k[0][2], eq[2][0] + eq[0][2], s20 + s02, w_zeta)
        diff = mixed(k[2][0] - k[0][2], eq[2][0] - eq[0][2], s20 - s02, w_nu)
        eq[1][1] = mixed(k[1][1], eq[1][1], s11, w_nu)
        eq[2][0], eq[0][2] = 0.5 * (both + diff), 0.5 * (both - diff)
        eq[0][0] = eq[0][0] + 0.5 * G
        eq[1][0] = eq[1][0] + 0.5 * (CS2 * Tx - ux * G)
        eq[0][1] = eq[0][1] + 0.5 * (CS2 * Ty - uy * G)
        self.g = self.streamed(_populations2(eq, ux, uy), rho)

    def streamed(self, a, rho=None):
        """Populations after streaming, with half-way bounce-back at walls (rho: the flow
        lattice, which the walls drag along)."""
        p = self.p
        out = [[None] * 3 for _ in range(3)]
        back = (0, 2, 1)
        for i, ex in enumerate(E1):
            for j, ey in enumerate(E1):
                v = torch.roll(a[i][j], (ey, ex), (0, 1)) if ex or ey else a[i][j].clone()
                if p.walls_y and ey:
                    row, u_wall = (0, -p.u_wall) if ey > 0 else (-1, p.u_wall)
                    v[row] = a[back[i]][back[j]][row]
                    if rho is not None:
                        v[row] += 2.0 * W1[i] * W1[j] * ex * u_wall * rho[row]
                out[i][j] = v
        return out


def _exact_fields(phys, fields, steps):
    s = _Exact2(phys, fields)
    for _ in range(steps):
        s.step()
    return s.macroscopic()


def _exact_diagnostics(phys, d):
    p, phi = phys, d["phi"]
    ny, nx = phi.shape
    X, Y = _grid(nx, ny)
    w = ((phi - p.phi_b) / (p.phi_a - p.phi_b)).clamp(0.0, 1.0)
    total = w.sum()

    def centre(at, n):
        t = 2.0 * math.pi / n * at
        return float(torch.atan2((w * torch.sin(t)).sum(), (w * torch.cos(t)).sum()) % (2.0 * math.pi)) * n / (2.0 * math.pi)

    xc = centre(X, nx)
    yc = float((w * Y).sum() / total) if p.walls_y else centre(Y, ny)
    dx = (X - xc + 0.5 * nx) % nx - 0.5 * nx
    dy = Y - yc if p.walls_y else (Y - yc + 0.5 * ny) % ny - 0.5 * ny
    xx, yy, xy = (float((w * v).sum() / total) for v in (dx * dx, dy * dy, dx * dy))
    half, root = 0.5 * (xx + yy), math.sqrt(max(0.25 * (xx - yy) ** 2 + xy * xy, 0.0))
    L, B = 4.0 * math.sqrt(half + root), 4.0 * math.sqrt(max(half - root, 0.0))
    found = {"sum_phi": float(phi.sum()), "sum_c": float(d["c"].sum()), "L": L, "B": B, "D": (L - B) / (L + B),
             "xc": xc, "yc": yc, "umax": float(torch.sqrt(d["ux"] ** 2 + d["uy"] ** 2).max())}
    found = {k: np.float64(v) for k, v in found.items()}
    found.update({k: None for k in ("step", "nonfinite", "sigma_neg", "status", "drops")})
    return found


def _exact3(case, seed):
    phi, c, u, W = _inputs_3d(case, seed)
    M, D = 0.05, 0.1
    zero = torch.zeros_like(phi)
    w3 = (1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0)

    def normal(v):
        def along(a, axis, weights):
            return sum(k * torch.roll(a, -e, axis) for e, k in zip((-1, 0, 1), weights) if k)
        d = (-0.5, 0.0, 0.5)  # 3 w1 e over the three offsets
        g = [along(along(along(v, 2, d if i == 0 else w3), 1, d if i == 1 else w3), 0, d if i == 2 else w3)
             for i in range(3)]
        m = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2)
        inv = torch.where(m > 1e-12, 1.0 / m, zero)
        return [x * inv for x in g]

    def collided(s, k):
        """Populations a[z][y][x] of central moments s mu mu mu and first moments k."""
        for zi, ez in enumerate(E1):
            Az, Bz, Cz = _from_central([1.0, 0.0, CS2], u[2])[zi], _from_central([0.0, 1.0, 0.0], u[2])[zi], \
                _from_central([1.0, 0.0, 0.0], u[2])[zi]
            for yi, ey in enumerate(E1):
                Ay, By, Cy = _from_central([1.0, 0.0, CS2], u[1])[yi], _from_central([0.0, 1.0, 0.0], u[1])[yi], \
                    _from_central([1.0, 0.0, 0.0], u[1])[yi]
                even, kx, ky = s * (Az * Ay), k[0] * (Cz * Cy), k[1] * (Cz * By) + k[2] * (Bz * Cy)
                for xi, ex in enumerate(E1):
                    Ax, Bx, Cx = _from_central([1.0, 0.0, CS2], u[0])[xi], _from_central([0.0, 1.0, 0.0], u[0])[xi], \
                        _from_central([1.0, 0.0, 0.0], u[0])[xi]
                    yield (ex, ey, ez), even * Ax + kx * Bx + ky * Cx

    def moments(pairs, stream_them):
        s, j = zero.clone(), [zero.clone() for _ in range(3)]
        for e, v in pairs:
            if stream_them:
                v = torch.roll(v, (e[2], e[1], e[0]), (0, 1, 2))
            s += v
            for i in range(3):
                if e[i]:
                    j[i] += e[i] * v
        return s, j

    n = normal(phi)
    theta = 4.0 / W * (1.0 - phi) * phi
    theta_c = 8.0 / W * c * (0.5 - phi)
    phi, jf = moments(collided(phi, [M * theta * x for x in n]), False)
    c, jh = moments(collided(c, [D * theta_c * x for x in n]), False)
    for _ in range(case["steps"]):
        n = normal(phi)
        theta = 4.0 / W * (1.0 - phi) * phi
        theta_c = 8.0 / W * c * (0.5 - phi)

        def relaxed(s, j, K, t):
            w = 1.0 / (3.0 * K + 0.5)
            k = [j[i] - u[i] * s for i in range(3)]
            return collided(s, [k[i] + w * (K * t * n[i] - k[i]) for i in range(3)])

        new = moments(relaxed(phi, jf, M, theta), True)
        c, jh = moments(relaxed(c, jh, D, theta_c), True)
        phi, jf = new
    return {"phi": phi, "c": c}


def _net_forward(params, X):
    a = X
    for l, (w, b) in enumerate(params):
        a = a @ w.to(torch.bfloat16).double().T + b
        if l < len(params) - 1:
            a = torch.nn.functional.silu(a)
    return a


def _net_params(net):
    return [[torch.from_numpy(w).cuda().double(), torch.from_numpy(b).cuda().double()] for w, b in net.get_params()]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "label"):
        phys, fields = _inputs_2d(case, seed)
        d = _exact_fields(phys, fields, case["steps"])
        if kind == "label":
            return _exact_diagnostics(phys, d)
        return {"phi": d["phi"], "c": d["c"], "u": torch.stack((d["ux"], d["uy"])), "P": d["P"]}
    if kind == "batch":
        got = [_exact_fields(phys, fields, case["steps"]) for phys, fields in _inputs_batch(case, seed)]
        return {"phi": torch.stack([d["phi"] for d in got]), "c": torch.stack([d["c"] for d in got]),
                "u": torch.stack([torch.stack((d["ux"], d["uy"])) for d in got]),
                "P": torch.stack([d["P"] for d in got])}
    if kind == "step3":
        return _exact3(case, seed)
    # the network's starting weights are the library's; everything after them is torch's
    net = lbm.Surrogate(seed=seed % 1000003)
    params = _net_params(net)
    net.close()
    data = _inputs_net(case, seed)
    if kind == "scan":
        out = _net_forward(params, torch.from_numpy(data).cuda().double())
        return {"D": out[:, 0], "logit": out[:, 1]}
    X, yD, yB = (torch.from_numpy(v).cuda().double() for v in data)

    def loss_of(at):
        out = _net_forward(at, X)
        return ((out[:, 0] - yD) ** 2).mean() + torch.nn.functional.binary_cross_entropy_with_logits(out[:, 1], yB)

    flat = [v for pair in params for v in pair]
    m, v2 = [torch.zeros_like(v) for v in flat], [torch.zeros_like(v) for v in flat]
    for t in range(1, case["epochs"] + 1):
        # the gradient at the rounded weights, applied to the unrounded ones
        at = [(w.to(torch.bfloat16).double().requires_grad_(), b.clone().requires_grad_())
              for w, b in zip(flat[::2], flat[1::2])]
        grads = torch.autograd.grad(loss_of(at), [v for pair in at for v in pair])
        for i, g in enumerate(grads):
            m[i] = 0.9 * m[i] + 0.1 * g
            v2[i] = 0.999 * v2[i] + 0.001 * g * g
            flat[i] = flat[i] - 2e-3 * (m[i] / (1.0 - 0.9 ** t)) / (torch.sqrt(v2[i] / (1.0 - 0.999 ** t)) + 1e-8)
    pairs = [[flat[2 * l], flat[2 * l + 1]] for l in range(len(flat) // 2)]
    return {"loss": loss_of(pairs).detach(), "params": pairs}
