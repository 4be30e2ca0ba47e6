"""The framework's work as a user's programs have it do, for timing and comparison.

A case is a lattice with its set-up, its precision and the number of lattice
steps of one pass.  ``prepare`` builds the initial fields on the GPU and the
simulation (or batch) that a program keeps; ``run`` advances it and reads the
fields back, as the measuring loops of the physics programs do.  Successive
passes go on from where the last one ended.

Set-ups follow the workloads of the package (static drop, capillary wave,
rising bubble, drop impact, Taylor bubble, batched sweep): lattice units,
heavy phase phi = 1, tanh interfaces, hydrostatic starts under gravity.  The
seed moves the interface by a fraction of a cell and draws a velocity noise
on top of the set-up's own flow.

Fields are returned in the precision a program keeps its snapshots in: FP64
for FP64 runs, FP32 for FP32 runs, FP16 for FP16S runs (whose stated accuracy
is 1e-3).
"""
import math

import numpy as np
import torch

from paper_2206_11637_gb300 import _lib as L
from paper_2206_11637_gb300 import workloads as W
from paper_2206_11637_gb300.batch import Batch
from paper_2206_11637_gb300.pflbm import Simulation

SNAPSHOT = {"fp64": torch.float64, "fp32": torch.float32, "fp16s": torch.float16}
POP_BYTES = {"fp64": 8, "fp32": 4, "fp16s": 2}


# ------------------------------------------------------------------ cases --

def listed():
    def c(name, kind, nx, ny, nz, precision, steps, lattice=15, count=1):
        return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
                "lattice": lattice, "count": count}

    return [
        # the smallest: a validation run in the reference precision (Laplace pressure, parity), few steps at a time
        c("drop_32_fp64", "drop", 32, 32, 32, "fp64", 10),
        # an odd lattice in the reference precision, as convergence checks against FP64 run
        c("bubble_61x183x61_fp64", "bubble", 61, 183, 61, "fp64", 4),
        # quasi-2-D waves: a small lattice stepped between two readings of the interface height
        c("wave_200x400_fp32", "wave", 200, 400, 1, "fp32", 100),
        c("wave_200x400_d2q9_fp16s", "wave", 200, 400, 1, "fp16s", 100, 9),
        # the rising bubble, the ordinary 3-D run, in both fast precisions and on the paper's own D3Q27 lattice
        c("bubble_128x384x128_fp32", "bubble", 128, 384, 128, "fp32", 32),
        c("bubble_128x384x128_fp16s", "bubble", 128, 384, 128, "fp16s", 32),
        c("bubble_128x384x128_d3q27_fp32", "bubble", 128, 384, 128, "fp32", 16, 27),
        # drop impacts: the half-size lattice, and the largest, which the benchmark runs
        c("impact_256x192x256_fp32", "impact", 256, 192, 256, "fp32", 40),
        c("impact_512x384x512_fp16s", "impact", 512, 384, 512, "fp16s", 40),
        # Taylor bubble in a voxelised tube (solid cells; the tube makes nx no multiple of a tile)
        c("taylor_66x640x66_fp32", "taylor", 66, 640, 66, "fp32", 32),
        # a parameter sweep: many uneven lattices, drops and waves, advanced together
        c("sweep_32_fp32", "sweep", 24, 96, 0, "fp32", 48, 15, 32),
        # the gradient of a match with an observed bubble with respect to mobility, interface width and surface tension
        c("adjoint_128x384x128_fp32", "adjoint", 128, 384, 128, "fp32", 25),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["drop", "wave", "bubble", "bubble", "impact", "impact", "taylor", "sweep", "adjoint"])
    precision = rng.choice(["fp64", "fp32", "fp32", "fp16s", "fp16s"])
    lattice, count = 15, 1
    if kind == "drop":
        nx = ny = nz = log(20, 160)
        lattice = rng.choice([15, 15, 27])
    elif kind == "wave":
        nx, nz = log(48, 600), 1
        ny = rng.choice([nx, 2 * nx])
        lattice = rng.choice([15, 9, 9])
    elif kind == "bubble":
        nx = log(32, 192)
        ny, nz = int(nx * rng.uniform(2.0, 3.0)), max(24, int(nx * rng.uniform(0.8, 1.2)))
        lattice = rng.choice([15, 15, 27])
    elif kind == "impact":
        nx = log(48, 330)
        ny, nz = int(nx * rng.uniform(0.7, 1.0)), int(nx * rng.uniform(0.8, 1.0))
    elif kind == "taylor":
        d = log(56, 96)  # narrower tubes at these numbers are unstable
        nx, ny, nz = d + 2, 10 * d, d + 2
    elif kind == "sweep":
        nx, ny, nz, count, precision = 24, log(40, 110), 0, log(4, 48), rng.choice(["fp32", "fp32", "fp32", "fp64"])
        count = min(count, 8) if precision == "fp64" else count
    else:
        nx = log(32, 128)
        ny, nz, precision = int(nx * rng.uniform(2.0, 3.0)), int(nx * rng.uniform(0.8, 1.0)), rng.choice(["fp32", "fp32", "fp64"])
    cells = nx * ny * max(nz, 1) if kind != "sweep" else count * ny ** 3 // 4
    steps = rng.randint(10, 48) if precision != "fp64" else rng.randint(2, max(2, min(16, int(4e7 / cells))))
    if kind == "adjoint":
        steps = rng.randint(4, 30) if precision != "fp64" else rng.randint(2, max(2, min(9, int(1e7 / cells))))
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps, "lattice": lattice,
            "count": count}


# ----------------------------------------------------------------- inputs --

def _axes(nx, ny, nz, dev):
    f = dict(dtype=torch.float64, device=dev)
    return (torch.arange(nx, **f).view(1, 1, nx), torch.arange(ny, **f).view(1, ny, 1), torch.arange(nz, **f).view(nz, 1, 1))


def _tanh(d, xi):
    return 0.5 - 0.5 * torch.tanh(d * (2.0 / xi))


def _hydrostatic(p, phi0, level, pressure=0.0, weight=None):
    """p* of the heavy fluid at rest, zero at y = level; `weight` blends a region of uniform pressure in."""
    _, y, _ = _axes(p.nx, p.ny, p.nz, phi0.device)
    pres = (p.rho_h * abs(p.gravity[1]) * (level - y)).expand(p.nz, p.ny, p.nx)
    if weight is not None:
        pres = (1.0 - weight) * pres + weight * pressure
    return 3.0 * pres / (p.rho_l + phi0 * (p.rho_h - p.rho_l))


def _one(kind, nx, ny, nz, lattice, seed, dev):
    """(params, phi0, u0, p0) of one lattice, fields as (nz, ny, nx) FP64 tensors on `dev`."""
    g = torch.Generator(device="cpu").manual_seed(int(seed))
    s = [2.0 * v - 1.0 for v in torch.rand(4, generator=g, dtype=torch.float64).tolist()]  # in (-1, 1)
    x, y, z = _axes(nx, ny, nz, dev)
    walls = (1,) * 6
    u_noise, uy, p0, solid, hydro, level = 1e-3, None, None, None, 0, 0.0
    if kind == "drop":
        p = W.Params(nx, ny, nz)
        r = ((x - (nx - 1) / 2 - s[0]) ** 2 + (y - (ny - 1) / 2 - s[1]) ** 2 + (z - (nz - 1) / 2 - s[2]) ** 2).sqrt()
        phi0 = _tanh(r - 0.3125 * nx, p.xi)
    elif kind == "wave":
        p = W.Params(nx, ny, nz, (0, 0, 1, 1, 0, 0), nu_h=0.01, nu_l=0.01)
        a0 = 0.01 * nx * (1.0 + 0.5 * s[0])
        ys = (ny - 1) / 2 + s[1] + a0 * torch.cos(2.0 * math.pi / nx * x)
        phi0 = _tanh((y - ys).expand(nz, ny, nx), p.xi)
    elif kind in ("bubble", "adjoint"):
        d, nu = nx / 4.0, 1.0 / 60.0
        grav = nu ** 2 * 10.0 ** 1.5 / (d ** 3 * math.sqrt(1e-3))
        p = W.Params(nx, ny, nz, walls, nu_h=nu, nu_l=10.0 * nu, sigma=grav * d * d / 10.0, xi=4.0, gravity=(0.0, -grav, 0.0))
        cy = 1.5 * d + s[1]
        r = ((x - (nx - 1) / 2 - s[0]) ** 2 + (y - cy) ** 2 + (z - (nz - 1) / 2 - s[2]) ** 2).sqrt()
        phi0 = _tanh(d / 2 - r, p.xi)
        p0 = _hydrostatic(p, phi0, cy, 2.0 * p.sigma / (d / 2), 1.0 - phi0)
    elif kind == "impact":
        d, depth, gap, speed = nx / 8.0, float(ny // 3), nx / 64.0, 0.05
        nu = (1.0 / 1.988 - 0.5) / 3.0
        p = W.Params(nx, ny, nz, walls, nu_h=nu, nu_l=20.0 * nu, sigma=speed ** 2 * d / 200.0, gravity=(0.0, -speed ** 2 / (200.0 * d), 0.0))
        cy = depth + gap + d / 2 + s[1]
        r = ((x - (nx - 1) / 2 - s[0]) ** 2 + (y - cy) ** 2 + (z - (nz - 1) / 2 - s[2]) ** 2).sqrt()
        drop, pool = _tanh(r - d / 2, p.xi), _tanh(y - depth, p.xi)
        phi0 = torch.maximum(drop, pool.expand_as(drop))
        uy = -speed * drop * (y > depth + gap / 2)
        pres = p.rho_h * abs(p.gravity[1]) * (depth - y).clamp(min=0.0) * pool + drop * (4.0 * p.sigma / d)
        p0 = 3.0 * pres / (p.rho_l + phi0 * (p.rho_h - p.rho_l))
        u_noise = 1e-4
    elif kind == "taylor":
        d, rho_ratio, mu_ratio = nx - 2, 744.0, 4236.0
        nu, rho_l = (1.0 / 1.76 - 0.5) / 3.0, 1.0 / rho_ratio
        sigma = nu ** 2 * math.sqrt(100.0 * (1.0 - rho_l) / 0.015) / d
        p = W.Params(nx, ny, nz, (0, 0, 1, 1, 0, 0), rho_l=rho_l, nu_h=nu, nu_l=nu * rho_ratio / mu_ratio, sigma=sigma,
                     mobility=0.08, xi=3.5, gravity=(0.0, -100.0 * sigma / (d * d), 0.0))
        r = ((x - (nx - 1) / 2) ** 2 + (z - (nz - 1) / 2) ** 2).sqrt()
        solid = (r > d / 2).expand(nz, ny, nx)
        yb, yt = d - 0.5 + s[0], 4 * d - 0.5 + s[1]
        phi0 = _tanh(-torch.maximum(r - 0.375 * d, torch.maximum(yb - y, y - yt)), p.xi)
        hydro, level = 1, yt  # the library's hydrostatic start
        u_noise = 1e-4
    p.h_lattice = lattice
    p.hydrostatic, p.p_level = hydro, level
    if solid is not None:
        p.solid = solid.to(torch.uint8).cpu().numpy()
    gd = torch.Generator(device=dev).manual_seed(int(seed))
    u0 = (2.0 * torch.rand((3, nz, ny, nx), generator=gd, dtype=torch.float64, device=dev) - 1.0) * u_noise
    if lattice == 9:
        u0[2] = 0.0
    if uy is not None:
        u0[1] += uy
    return p, phi0.contiguous(), u0, None if p0 is None else p0.contiguous()


def _sweep_sizes(case):
    """Sizes of a sweep's instances, fixed by the case: cubes (with a drop) and quasi-2-D lattices (with a wave) in turn."""
    rng = np.random.Generator(np.random.PCG64(case["count"] * 1000 + case["ny"]))
    out = []
    for i in range(case["count"]):
        n = int(rng.integers(case["nx"], case["ny"] + 1)) * (1 if i % 2 == 0 else 2)
        out.append((n, n, n) if i % 2 == 0 else (n, 2 * n, 1))
    return out


def _sweep(case, seed, dev):
    """The instances of a sweep, M and sigma drawn from the seed."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    out = []
    for i, (nx, ny, nz) in enumerate(_sweep_sizes(case)):
        q = _one("wave" if nz == 1 else "drop", nx, ny, nz, 15, seed + i, dev)
        q[0].mobility, q[0].sigma = float(rng.uniform(0.005, 0.1)), float(10.0 ** rng.uniform(-5.0, -3.0))
        out.append(q)
    return out


def _inputs(case, seed, dev="cuda"):
    if case["kind"] == "sweep":
        return _sweep(case, seed, dev)
    return [_one(case["kind"], case["nx"], case["ny"], case["nz"], case["lattice"], seed, dev)]


def _match_weights(case, dev="cuda"):
    """J: the overlap of phi with an observed bubble one cell higher, at half the horizon and at its end, as weights of phi."""
    nx, ny, nz, n = case["nx"], case["ny"], case["nz"], case["steps"]
    x, y, z = _axes(nx, ny, nz, dev)
    r = ((x - (nx - 1) / 2) ** 2 + (y - 0.375 * nx - 1.0) ** 2 + (z - (nz - 1) / 2) ** 2).sqrt()
    w = _tanh(nx / 8.0 - r, 4.0) / float(nx * ny * nz)
    return [(n // 2, w), (n, w.clone())]


def prepare(case, seed):
    if case["kind"] == "sweep":
        inst = [(p, phi0.cpu().numpy(), u0.cpu().numpy(), None) for p, phi0, u0, _ in _inputs(case, seed)]
        b = Batch(inst, precision=case["precision"])
        out = [{"phi": torch.empty(q[0].shape, dtype=torch.float64, device="cuda"),
                "u": torch.empty((3,) + q[0].shape, dtype=torch.float64, device="cuda")} for q in inst]
        return {"case": case, "batch": b, "out": out}
    p, phi0, u0, p0 = _inputs(case, seed)[0]
    sim = Simulation(p, phi0, u0, p0, precision=case["precision"])
    if case["kind"] == "adjoint":
        return {"case": case, "sim": sim, "obs": [(k, w.view(-1)) for k, w in _match_weights(case)]}
    names = ("phi", "rho", "p", "u") if case["precision"] == "fp64" else ("phi", "u")
    out = {k: torch.empty(((3,) if k == "u" else ()) + p.shape, dtype=torch.float64, device="cuda") for k in names}
    return {"case": case, "sim": sim, "out": out}


def run(state):
    case = state["case"]
    keep = SNAPSHOT[case["precision"]]
    if case["kind"] == "sweep":
        b = state["batch"]
        b.step(case["steps"])
        for i, o in enumerate(state["out"]):  # into device arrays, through the C interface
            L.check(b.lib.pfl_batch_fields(b.b, i, o["phi"].data_ptr(), None, None, o["u"].data_ptr()))
        return {k: torch.cat([o[k].view(-1) for o in state["out"]]).to(keep) for k in ("phi", "u")}
    sim = state["sim"]
    if case["kind"] == "adjoint":
        J, grad = sim.adjoint(case["steps"], state["obs"])
        return {"J": torch.tensor(J, dtype=keep), "grad": torch.from_numpy(grad).to(keep)}
    sim.step(case["steps"])
    out = sim.fields(out=state["out"])
    res = {k: v.to(keep) for k, v in out.items()}
    if case["kind"] == "wave":
        res["height"] = torch.tensor(sim.interface_height(0, 0), dtype=torch.float32)
    return res


def work(case):
    """Per lattice step every population is read once and written once and phi written; a pass also reads g and phi
    once and writes the fields.  An adjoint step reads the state and lambda and writes lambda (the forward sweep
    reads and writes the state).  Operations: additions and multiplications of the closed-form update, about 10 per
    population, and of its reverse."""
    s = POP_BYTES[case["precision"]]
    r = 8 if case["precision"] == "fp64" else 4
    qh = case["lattice"]
    qg = 9 if qh == 9 else 27
    if case["kind"] == "sweep":
        cells = float(sum(nx * ny * nz for nx, ny, nz in _sweep_sizes(case)))
    else:
        cells = float(case["nx"] * case["ny"] * case["nz"])
    step = 2 * (qh + qg) * s + r + (8 if case["precision"] == "fp16s" else 0)
    n = case["steps"]
    if case["kind"] == "adjoint":
        return {"bytes": cells * n * (step + (qh + qg) * (s + 2 * r)), "flops": cells * n * 30.0 * (qh + qg)}
    fields = 6 if case["precision"] == "fp64" else 4
    return {"bytes": cells * (n * step + qg * s + r + 8 * fields), "flops": cells * n * 10.0 * (qh + qg)}


# -------------------------------------------------- the same in 64 bits ----
# The update written out in plain torch: moments, forces and the
# weighted-orthogonal MRT collision in closed form, push streaming with
# half-way bounce-back, phi = sum h.

class _Exact:
    def __init__(self, p, lattice, dev):
        self.p, self.dev, self.lattice = p, dev, lattice
        c27 = [(cx, cy, cz) for cz in (-1, 0, 1) for cy in (-1, 0, 1) for cx in (-1, 0, 1)]
        w27 = {0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216}
        w15 = {0: 2 / 9, 1: 1 / 9, 3: 1 / 72}
        w9 = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
        n2 = lambda c: c[0] ** 2 + c[1] ** 2 + c[2] ** 2  # noqa: E731
        c9 = [c for c in c27 if c[2] == 0]
        self.gl = [(c, w9[n2(c)]) for c in c9] if lattice == 9 else [(c, w27[n2(c)]) for c in c27]
        self.hl = {15: [(c, w15[n2(c)]) for c in c27 if n2(c) in w15], 27: [(c, w27[n2(c)]) for c in c27],
                   9: [(c, w9[n2(c)]) for c in c9]}[lattice]
        self.trace = 2 if lattice == 9 else 3
        self.wall = [p.bc[0] == 1, p.bc[2] == 1, p.bc[4] == 1]
        solid = getattr(p, "solid", None)
        self.solid = None if solid is None else torch.from_numpy(np.ascontiguousarray(solid)).to(dev).reshape(p.shape) != 0
        self.blocked = {}
        n = (p.nx, p.ny, p.nz)
        for c in {c for c, _ in self.gl}:  # cells whose source x - c lies behind a wall or in a solid
            m = None
            for a in range(3):
                if c[a] and self.wall[a]:
                    i = torch.arange(n[a], device=dev)
                    e = ((i == 0) if c[a] > 0 else (i == n[a] - 1)).view([-1 if 2 - a == k else 1 for k in range(3)])
                    m = e if m is None else m | e
            if self.solid is not None and any(c):
                b = torch.roll(self.solid, (c[2], c[1], c[0]), (0, 1, 2))
                m = b if m is None else m | b
            self.blocked[c] = m

    def at(self, f, c):
        """f at x + c, mirrored at walls and solids as the stencil reads it."""
        v = f
        n = (self.p.nx, self.p.ny, self.p.nz)
        for a in range(3):
            if c[a]:
                i = torch.arange(n[a], device=self.dev) + c[a]
                i = i.clamp(0, n[a] - 1) if self.wall[a] else i % n[a]
                v = v.index_select(2 - a, i)
        if self.solid is not None and any(c):
            v = torch.where(torch.roll(self.solid, (-c[2], -c[1], -c[0]), (0, 1, 2)), f, v)
        return v

    def stream(self, post, lat):
        idx = {c: k for k, (c, _) in enumerate(lat)}
        new = []
        for k, (c, _) in enumerate(lat):
            f = torch.roll(post[k], (c[2], c[1], c[0]), (0, 1, 2)) if any(c) else post[k]
            if self.blocked[c] is not None:
                f = torch.where(self.blocked[c], post[idx[(-c[0], -c[1], -c[2])]], f)
            if self.solid is not None:
                f = torch.where(self.solid, torch.zeros_like(f), f)
            new.append(f)
        return new

    def start(self, phi0, u0, p0):
        u = u0
        if p0 is None:
            p0 = torch.zeros_like(phi0)
        if self.p.hydrostatic:  # dp/dy = rho g by the trapezoid rule, zero at y = p_level
            rho = self.p.rho_l + phi0 * (self.p.rho_h - self.p.rho_l)
            P = torch.cumsum(0.5 * (rho[:, 1:] + rho[:, :-1]), 1) * self.p.gravity[1]
            P = torch.cat([torch.zeros_like(P[:, :1]), P], 1)
            j = min(max(int(math.floor(self.p.p_level)), 0), self.p.ny - 2)
            t = self.p.p_level - j
            P = P - ((1 - t) * P[:, j:j + 1] + t * P[:, j + 1:j + 2])
            p0 = 3.0 * P / rho
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        h, g = [], []
        for c, w in self.hl:
            h.append(w * phi0 * (1 + 3 * (c[0] * u[0] + c[1] * u[1] + c[2] * u[2])))
        for c, w in self.gl:
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            g.append(w * (p0 + 3 * cu + 4.5 * cu * cu - 1.5 * uu))
        if self.solid is not None:
            h = [torch.where(self.solid, torch.zeros_like(f), f) for f in h]
            g = [torch.where(self.solid, torch.zeros_like(f), f) for f in g]
        return h, g

    def macro(self, h, g, M, xi, sigma):
        p = self.p
        phi = sum(h)
        G = [0.0, 0.0, 0.0]
        lap = 0.0
        for c, w in self.gl:
            if any(c):
                d = self.at(phi, c) - phi
                lap = lap + 6 * w * d
                for a in range(3):
                    if c[a]:
                        G[a] = G[a] + 3 * w * c[a] * d
        if self.lattice == 9:
            G[2] = torch.zeros_like(phi)
        ps = sum(g)
        j = [sum(c[a] * f for (c, _), f in zip(self.gl, g) if c[a]) if any(c[a] for c, _ in self.gl) else torch.zeros_like(phi)
             for a in range(3)]
        second = lambda lat, f, a, b: sum(  # noqa: E731
            (c[a] * c[b] * v for (c, _), v in zip(lat, f) if c[a] * c[b]), torch.zeros_like(phi))
        P = {(a, b): second(self.gl, g, a, b) for a in range(3) for b in range(a, 3)}
        drho = p.rho_h - p.rho_l
        rho = p.rho_l + phi * drho
        tau_h, tau_l = 3 * p.nu_h + 0.5, 3 * p.nu_l + 0.5
        tau = tau_l + phi * (tau_h - tau_l)
        omega, nu = 1 / tau, (tau - 0.5) / 3
        mu = 4 * (12 * sigma / xi) * phi * (phi - 1) * (phi - 0.5) - 1.5 * sigma * xi * lap
        F = [(mu - ps * drho / 3) * G[a] + rho * p.gravity[a] for a in range(3)]
        u0 = [j[a] + F[a] / (2 * rho) for a in range(3)]
        N = {(a, b): P[a, b] - (ps / 3 if a == b else 0) - u0[a] * u0[b] for a, b in P}
        cm = -3 * nu * omega * drho
        F = [F[a] + cm * sum(N[min(a, b), max(a, b)] * G[b] for b in range(3)) for a in range(3)]
        u = [j[a] + F[a] / (2 * rho) for a in range(3)]
        return phi, rho, ps, u, F, G, P, omega

    def step(self, h, g, M, xi, sigma):
        phi, rho, ps, u, F, G, P, omega = self.macro(h, g, M, xi, sigma)
        T = range(self.trace)
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        a2 = 4.5 * (1 - omega)
        D = {(a, b): P[a, b] - (ps / 3 if a == b else 0) - u[a] * u[b] for a, b in P}
        tr = sum(D[a, a] for a in T) / 3
        post = []
        for c, w in self.gl:
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            cf = 1.5 * (c[0] * F[0] + c[1] * F[1] + c[2] * F[2]) / rho
            cc = sum((1 if a == b else 2) * c[a] * c[b] * D[a, b] for a, b in D if c[a] * c[b]) if any(c) else 0.0
            post.append(w * (ps + 3 * cu + 4.5 * cu * cu - 1.5 * uu + a2 * (cc - tr) + cf))
        g2 = self.stream(post, self.gl)
        del post
        om = 1 / (3 * M + 0.5)
        j = [sum((c[a] * f for (c, _), f in zip(self.hl, h) if c[a]), torch.zeros_like(phi)) for a in range(3)]
        H = {(a, b): sum((c[a] * c[b] * f for (c, _), f in zip(self.hl, h) if c[a] * c[b]), torch.zeros_like(phi))
             - (phi / 3 if a == b else 0) for a in range(3) for b in range(a, 3)}
        tr = sum(H[a, a] for a in T) / 3
        sq = G[0] ** 2 + G[1] ** 2 + G[2] ** 2
        gn = torch.where(sq > 0, torch.where(sq > 0, sq, torch.ones_like(sq)).sqrt(), torch.zeros_like(sq))
        tn = 4 * phi * (1 - phi) / xi / (gn + 1e-6) * (1 - 0.5 * om)
        beta = [3 * phi * u[a] + 3 * (1 - om) * (j[a] - phi * u[a]) + tn * G[a] for a in range(3)]
        b2 = 4.5 * (1 - om)
        post = []
        for c, w in self.hl:
            cc = sum((1 if a == b else 2) * c[a] * c[b] * H[a, b] for a, b in H if c[a] * c[b]) if any(c) else 0.0
            post.append(w * (phi + c[0] * beta[0] + c[1] * beta[1] + c[2] * beta[2] + b2 * (cc - tr)))
        return self.stream(post, self.hl), g2


def exact(case, seed):
    with torch.no_grad():
        inst = _inputs(case, seed)
    if case["kind"] == "adjoint":
        return _exact_gradient(case, inst[0])
    res = []
    with torch.no_grad():
        for p, phi0, u0, p0 in inst:
            e = _Exact(p, case["lattice"], phi0.device)
            h, g = e.start(phi0, u0, p0)
            del phi0, u0, p0
            for _ in range(case["steps"]):
                h, g = e.step(h, g, p.mobility, p.xi, p.sigma)
            phi, rho, ps, u, *_ = e.macro(h, g, p.mobility, p.xi, p.sigma)
            del h, g
            fluid = 1.0 if e.solid is None else (~e.solid).double()
            res.append({"phi": phi * fluid, "rho": rho * fluid, "p": ps * rho / 3 * fluid,
                        "u": torch.stack(u) * fluid})
    if case["kind"] == "sweep":
        return {k: torch.cat([o[k].view(-1) for o in res]) for k in ("phi", "u")}
    out = res[0] if case["precision"] == "fp64" else {k: res[0][k] for k in ("phi", "u")}
    if case["kind"] == "wave":  # first phi = 1/2 crossing of the column x = 0 from the heavy side
        col = out["phi"][0, :, 0]
        k = int(((col[:-1] >= 0.5) & (col[1:] < 0.5)).nonzero()[0])
        out["height"] = float(k + (col[k] - 0.5) / (col[k] - col[k + 1]))
    return out


def _exact_gradient(case, q):
    from torch.utils.checkpoint import checkpoint
    p, phi0, u0, p0 = q
    dev = phi0.device
    par = [torch.tensor(v, dtype=torch.float64, device=dev, requires_grad=True) for v in (p.mobility, p.xi, p.sigma)]
    e = _Exact(p, case["lattice"], dev)
    with torch.no_grad():
        h, g = e.start(phi0, u0, p0)
    nh = len(h)

    def one(M, xi, sigma, *f):
        a, b = e.step(list(f[:nh]), list(f[nh:]), M, xi, sigma)
        return tuple(a) + tuple(b)

    obs = dict(_match_weights(case))
    J = 0.0
    f = tuple(h) + tuple(g)
    for k in range(case["steps"] + 1):
        if k in obs:
            J = J + (obs[k] * sum(f[:nh])).sum()
        if k < case["steps"]:
            f = checkpoint(one, *par, *f, use_reentrant=False)
    grad = torch.autograd.grad(J, par)
    return {"J": J.detach(), "grad": torch.stack(list(grad)).detach()}
