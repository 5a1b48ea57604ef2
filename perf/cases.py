"""The work that users have this framework do, as measurable cases.

A case is one whole job through the public classes: hand over an initial field,
advance the time steps, read the result (for the adjoint: a forward run and its
gradients). Five kinds, told apart by case["kind"]:

  grid      one D2Q9 lattice, Scheme B (Solver): FP64, FP32 or BF16-shifted
            storage, periodic or anti-bounce-back walls, constant or per-node K
  general   one D2Q9 lattice on the general path (Solver): Scheme A, power-law
            flux, Fisher source, extrapolated walls with time-dependent values
  ensemble  many independent D2Q9 lattices of different sizes (Ensemble)
  adjoint   a differentiable run and its gradients in phi0, K(x) and u (adjoint)
  grid3     one D3Q19 lattice (Solver3)

listed() gives twelve of them, draw(rng) more of the same ranges, prepare() what a
program holds before the call, run() one job, work() the bytes and operations a job
cannot do without, and exact() the same job in 64-bit torch operations, written from
the equations without this package.
"""
import math
import random

import numpy as np
import torch

# relaxation rates s0..s8 of the moments; entries 3 and 5 come from the tensor K
RATES = (1.0, 1.2, 1.2, 0.0, 1.0, 0.0, 1.0, 1.1, 1.1)
# the launch that the autotuner keeps for FP32 and BF16S on large grids, and the
# constructor's own defaults
TUNED = dict(spp=2, variant=5, rows=4)
DEFAULT = dict(spp=1, variant=0, rows=0)
TWO = dict(spp=2, variant=0, rows=0)


def listed():
    return [
        # the paper's isotropic Gaussian hill in double precision: the smallest grid that
        # people run, for convergence tables, with the error norms read at the end
        dict(name="gaussian_128_f64", kind="grid", nx=128, ny=128, prec="f64", bcx="periodic", bcy="periodic",
             conv=0, ux=0.05, uy=0.02, diff=0, kxx=0.01, kxy=0.0, kyy=0.01, r1=0.0, field="hill", stats=True,
             steps=1000, cellk=False, **DEFAULT),
        # the paper's anisotropic 400^2 hill as a first program has it: FP32, every argument of
        # the constructor left at its default, many steps of a small grid
        dict(name="hill_400_f32", kind="grid", nx=400, ny=400, prec="f32", bcx="periodic", bcy="periodic",
             conv=0, ux=0.01, uy=0.01, diff=0, kxx=0.2, kxy=0.2, kyy=0.4, r1=0.0, field="hill", stats=False,
             steps=1000, cellk=False, **DEFAULT),
        # a ragged grid with walls on one axis, nonlinear flux, diffusion and source, an odd
        # number of steps, two steps per pass asked for and the rest left automatic
        dict(name="ragged_1023x777_f32", kind="grid", nx=1023, ny=777, prec="f32", bcx="abb", bcy="periodic",
             conv=1, ux=0.08, uy=-0.05, diff=1, kxx=0.02, kxy=0.008, kyy=0.01, r1=-0.0005, field="noise", stats=False,
             steps=251, cellk=False, **TWO),
        # the Burgers workload on its 1024^2 grid, autotuned launch
        dict(name="burgers_1024_f32", kind="grid", nx=1024, ny=1024, prec="f32", bcx="periodic", bcy="periodic",
             conv=1, ux=math.sqrt(0.5), uy=math.sqrt(0.5), diff=0, kxx=5.12, kxy=0.0, kyy=5.12, r1=0.0, field="sine",
             stats=False, steps=500, cellk=False, **TUNED),
        # the headline: 4096^2 anisotropic nonlinear diffusion between walls, FP32
        dict(name="dirichlet_4096_f32", kind="grid", nx=4096, ny=4096, prec="f32", bcx="abb", bcy="abb",
             conv=0, ux=0.0, uy=0.0, diff=2, kxx=0.02, kxy=0.008, kyy=0.01, r1=-0.00005, field="noise", stats=False,
             steps=100, cellk=False, **TUNED),
        # the same in BF16-shifted storage, for the largest grids that fit
        dict(name="dirichlet_4096_bf16s", kind="grid", nx=4096, ny=4096, prec="bf16s", bcx="abb", bcy="abb",
             conv=0, ux=0.0, uy=0.0, diff=2, kxx=0.02, kxy=0.008, kyy=0.01, r1=-0.00005, field="noise", stats=False,
             steps=100, cellk=False, **TUNED),
        # a reference solution in double precision on a large grid
        dict(name="dirichlet_2048_f64", kind="grid", nx=2048, ny=2048, prec="f64", bcx="abb", bcy="abb",
             conv=0, ux=0.0, uy=0.0, diff=2, kxx=0.02, kxy=0.008, kyy=0.01, r1=-0.00005, field="noise", stats=True,
             steps=20, cellk=False, **DEFAULT),
        # the Burgers-Fisher problem on the paper's 301^2 nodes, Dirichlet values of every step
        dict(name="burgers_fisher_301_f32", kind="general", n=301, prec="f32", spp=2, steps=400),
        # gradients of a misfit in the tensor field, the drift and the initial field, 512^2
        dict(name="adjoint_512_f32", kind="adjoint", nx=512, ny=512, prec="f32", steps=500, every=50),
        # a parameter study: 128 lattices of 64 to 1024 nodes a side advanced together
        dict(name="ensemble_128", kind="ensemble", count=128, small=64, large=1024, sizes=5, spp=2, steps=100),
        # the 3-D Gaussian hill with a full tensor, 256^3
        dict(name="gaussian3d_256_f32", kind="grid3", nx=256, ny=256, nz=256, prec="f32", bcx="periodic",
             bcy="periodic", bcz="periodic", conv=0, diff=0, r1=0.0, steps=40),
        # a ragged 3-D channel between two walls in BF16-shifted storage
        dict(name="channel3d_201_bf16s", kind="grid3", nx=201, ny=130, nz=97, prec="bf16s", bcx="periodic",
             bcy="abb", bcz="periodic", conv=1, diff=1, r1=-0.0005, steps=60),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid"] * 7 + ["general"] * 2 + ["ensemble", "adjoint"] + ["grid3"] * 3)
    if kind == "grid":
        prec = rng.choice(["f32", "f32", "f32", "bf16s", "f64"])
        top = 2048 if prec == "f64" else 4096
        nx = _log_int(rng, 48, top)
        ny = max(16, min(top, int(nx * math.exp(rng.uniform(-0.7, 0.7)))))
        budget = 8e7 if prec == "f64" else 1.2e9
        steps = max(1, min(_log_int(rng, 10, 1000), int(budget / (nx * ny))))
        launch = DEFAULT if prec == "f64" else rng.choice([DEFAULT, TWO, TUNED])
        conv = rng.choice([0, 0, 1])
        drift = rng.choice([0.0, 0.04, 0.08])
        return dict(kind=kind, nx=nx, ny=ny, prec=prec, bcx=rng.choice(["periodic", "abb"]),
                    bcy=rng.choice(["periodic", "abb"]), conv=conv, ux=drift, uy=-0.6 * drift, diff=rng.choice([0, 1, 2]),
                    kxx=0.02, kxy=rng.choice([0.0, 0.008]), kyy=0.015, r1=rng.choice([0.0, -0.0005]),
                    field=rng.choice(["hill", "noise", "noise"]), stats=prec == "f64", steps=steps,
                    cellk=rng.random() < 0.2, **launch)
    if kind == "general":
        prec = rng.choice(["f32", "f32", "f64"])
        n = _log_int(rng, 60, 600 if prec == "f64" else 1500)
        return dict(kind=kind, n=n, prec=prec, spp=1 if prec == "f64" else rng.choice([1, 2]),
                    steps=min(_log_int(rng, 20, 600), int((4e7 if prec == "f64" else 2e8) / (n * n))))
    if kind == "ensemble":
        return dict(kind=kind, count=_log_int(rng, 8, 90), small=_log_int(rng, 40, 120), large=_log_int(rng, 200, 1000),
                    sizes=rng.randrange(1 << 20), spp=rng.choice([1, 2, 2]), steps=_log_int(rng, 20, 100))
    if kind == "adjoint":
        return dict(kind=kind, nx=_log_int(rng, 64, 512), ny=_log_int(rng, 64, 512), prec=rng.choice(["f32", "f32", "f64"]),
                    steps=_log_int(rng, 40, 300), every=rng.choice([20, 50]))
    prec = rng.choice(["f32", "f32", "bf16s", "f64"])
    top = 100 if prec == "f64" else 256
    nx, ny, nz = (_log_int(rng, 24, top) for _ in range(3))
    budget = 1.2e7 if prec == "f64" else 5e8
    return dict(kind="grid3", nx=nx, ny=ny, nz=nz, prec=prec, bcx=rng.choice(["periodic", "periodic", "abb"]),
                bcy=rng.choice(["periodic", "abb"]), bcz=rng.choice(["periodic", "periodic", "abb"]),
                conv=rng.choice([0, 1]), diff=rng.choice([0, 1, 2]), r1=rng.choice([0.0, -0.0005]),
                steps=max(1, min(_log_int(rng, 8, 200), int(budget / (nx * ny * nz)))))


# ---- inputs, from the seed alone -------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _real(prec):
    return torch.float64 if prec == "f64" else torch.float32


def _hill(nx, ny, xc, yc, sigma, amp):
    """Periodic Gaussian hill (nearest-image distance), FP64."""
    x = torch.arange(nx, device="cuda", dtype=torch.float64)
    y = torch.arange(ny, device="cuda", dtype=torch.float64)
    dx = (x - xc + nx / 2) % nx - nx / 2
    dy = (y - yc + ny / 2) % ny - ny / 2
    return amp * torch.exp(-(dy[:, None] ** 2 + dx[None, :] ** 2) / (2.0 * sigma * sigma))


def _noise(nx, ny, g):
    """U[0, 1) smoothed by three passes of the mean of the four neighbours, zero outside."""
    a = torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float64)
    for _ in range(3):
        p = torch.nn.functional.pad(a, (1, 1, 1, 1))
        a = 0.25 * (p[:-2, 1:-1] + p[2:, 1:-1] + p[1:-1, :-2] + p[1:-1, 2:])
    return a


def _smooth(nx, ny, rng):
    """A sum of eight random periodic Fourier modes, |k| <= 4, scaled to unit maximum."""
    x = torch.arange(nx, device="cuda", dtype=torch.float64) / nx
    y = torch.arange(ny, device="cuda", dtype=torch.float64) / ny
    f = torch.zeros((ny, nx), device="cuda", dtype=torch.float64)
    for _ in range(8):
        kx, ky = rng.randint(-4, 4), rng.randint(-4, 4)
        if kx == 0 and ky == 0:
            kx = 1
        f += rng.gauss(0, 1) * torch.cos(2 * math.pi * (kx * x[None, :] + ky * y[:, None]) + rng.uniform(0, 2 * math.pi))
    return f / f.abs().max()


def _tensor_field(nx, ny, rng):
    """A smooth symmetric positive definite tensor field (3, ny, nx): Kxx, Kxy, Kyy."""
    kxx = 0.005 + 0.045 * torch.sigmoid(2.0 * _smooth(nx, ny, rng))
    kyy = 0.005 + 0.045 * torch.sigmoid(2.0 * _smooth(nx, ny, rng))
    kxy = 0.5 * torch.sqrt(kxx * kyy) * torch.tanh(_smooth(nx, ny, rng))
    return torch.stack([kxx, kxy, kyy])


def _grid_inputs(c, seed):
    g, rng, nx, ny = _gen(seed), random.Random(seed), c["nx"], c["ny"]
    if c["field"] == "hill":
        phi = _hill(nx, ny, rng.uniform(0.3, 0.7) * nx, rng.uniform(0.3, 0.7) * ny,
                    max(4.0, rng.uniform(1 / 20, 1 / 12) * min(nx, ny)), rng.uniform(0.5, 1.0))
    elif c["field"] == "sine":
        x = torch.arange(nx, device="cuda", dtype=torch.float64) / nx
        y = torch.arange(ny, device="cuda", dtype=torch.float64) / ny
        phi = 0.5 * torch.sin(2 * math.pi * x)[None, :] * torch.sin(2 * math.pi * y)[:, None]
        phi = phi + 1e-3 * (2 * torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float64) - 1)
    else:
        phi = _noise(nx, ny, g)
    walls = tuple(rng.uniform(0.0, 0.4) for _ in range(4))
    K = _tensor_field(nx, ny, rng) if c["cellk"] else None
    return dict(phi=phi.to(_real(c["prec"])).contiguous(), walls=walls, K=K)


def _fisher_inputs(c, seed):
    """Burgers-Fisher travelling wave on [-1, 2]^2 (a = 4, b = 1, kappa = 0.12, delta = 1,
    dx/dt = 40): the initial field and the wall values of every step, FP64."""
    rng, n, steps = random.Random(seed), c["n"], c["steps"]
    a, b, kappa, speed = 4.0, 1.0, 0.12, 40.0
    off = rng.uniform(-0.4, 0.4)
    dx = 3.0 / (n - 1)
    dt = dx / speed
    w = (a * a + 8.0 * b * kappa) / (2.0 * a)
    xs = -1.0 + dx * torch.arange(n, device="cuda", dtype=torch.float64)

    def wave(x, y, t):
        return 0.5 + 0.5 * torch.tanh(-a / (8.0 * kappa) * (x + y - off - w * t))

    t = dt * torch.arange(1, steps + 1, device="cuda", dtype=torch.float64)[:, None]
    rec = torch.cat([wave(xs[0], xs[None, :], t), wave(xs[-1], xs[None, :], t),
                     wave(xs[None, :], xs[0], t), wave(xs[None, :], xs[-1], t)], 1)
    phi = wave(xs[None, :], xs[:, None], 0.0)
    return dict(phi=phi.to(_real(c["prec"])).contiguous(), rec=rec.contiguous(), ax=a * dt / dx, b=b * dt,
                K=kappa * dt / dx ** 2)


def _sides(c):
    """The lattices' sides, log-uniform between the smallest and the largest (part of the case, not of the inputs)."""
    rng = random.Random(c["sizes"])
    return [_log_int(rng, c["small"], c["large"]) for _ in range(c["count"])]


def _ensemble_inputs(c, seed):
    """Per lattice: drift |u| <= 0.1, diffusivity 0.001 to 0.05, the rates that keep such pairs
    stable ((1/s_odd - 1/2)(1/s_even - 1/2) = 1/4), and a Gaussian hill."""
    rng, inst, fields = random.Random(seed), [], []
    for n in _sides(c):
        r, th = 0.1 * math.sqrt(rng.random()), rng.uniform(0, 2 * math.pi)
        d0 = rng.uniform(0.001, 0.05)
        odd, even = 1.0 / (0.5 + 3.0 * d0), 1.0 / (0.5 + 0.25 / (3.0 * d0))
        inst.append(dict(nx=n, ny=n, u=(r * math.cos(th), r * math.sin(th)), K=(d0, 0.0, d0),
                         s=(1.0, even, even, 0.0, odd, 0.0, odd, even, even)))
        fields.append(_hill(n, n, rng.uniform(0, n), rng.uniform(0, n), max(4.0, rng.uniform(n / 32, n / 8)),
                            rng.uniform(0.5, 1.0)).float())
    return inst, fields


def _adjoint_inputs(c, seed):
    """Parameters to be fitted (the tensor field, the drift, the initial field) and a target."""
    rng, nx, ny = random.Random(seed), c["nx"], c["ny"]
    dt = _real(c["prec"])
    K = _tensor_field(nx, ny, rng).to(dt)
    phi = (0.5 + 0.4 * _smooth(nx, ny, rng)).to(dt)
    target = (0.5 + 0.4 * _smooth(nx, ny, rng)).to(dt)
    u = torch.tensor([0.03, rng.uniform(-0.01, 0.01)], dtype=dt, device="cuda")
    return phi, K, u, target


def _grid3_inputs(c, seed):
    rng, n = random.Random(seed), (c["nz"], c["ny"], c["nx"])
    ax = [torch.arange(m, device="cuda", dtype=torch.float64) - rng.uniform(0.4, 0.6) * m for m in n]
    s = max(3.0, min(n) / 16.0)
    phi = 0.1 + torch.exp(-(ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2][None, None, :] ** 2) / (2 * s * s))
    phi = phi + 0.01 * torch.rand(n, generator=_gen(seed), device="cuda", dtype=torch.float64)
    return dict(phi=phi.to(_real(c["prec"])).contiguous(), walls=tuple(rng.uniform(0.0, 0.4) for _ in range(6)))


K3 = (0.02, 0.006, 0.004, 0.015, 0.003, 0.01)       # xx, xy, xz, yy, yz, zz
SE3 = 1.1
U3 = {0: (0.02, 0.01, -0.015), 1: (0.05, -0.03, 0.02)}


def prepare(case, seed):
    from paper_1603_09577_gb300 import Ensemble, Solver, Solver3
    c, kind = case, case["kind"]
    if kind == "grid":
        d = _grid_inputs(c, seed)
        s = Solver(c["nx"], c["ny"], prec=c["prec"], bc=(c["bcx"], c["bcy"]), phi_wall=d["walls"],
                   steps_per_pass=c["spp"], kernel_variant=c["variant"], block_rows=c["rows"], per_cell_K=c["cellk"])
        s.set_coeffs(conv=c["conv"], u=(c["ux"], c["uy"]), diff=c["diff"], K=(c["kxx"], c["kxy"], c["kyy"]), s=RATES,
                     r1=c["r1"])
        if c["cellk"]:
            s.set_K_field(d["K"])
        return dict(c=c, s=s, phi=d["phi"])
    if kind == "general":
        d = _fisher_inputs(c, seed)
        s = Solver(c["n"], c["n"], prec=c["prec"], bc=("nee", "nee"), scheme="A", steps_per_pass=c["spp"])
        s.set_coeffs(conv=2, power=1, u=(d["ax"], 0.0), diff=0, K=(d["K"], 0.0, d["K"]), s=RATES, src_family=1, b=d["b"])
        s.set_dirichlet(d["rec"])
        return dict(c=c, s=s, phi=d["phi"])
    if kind == "ensemble":
        inst, fields = _ensemble_inputs(c, seed)
        e = Ensemble(inst, conv=0, diff=1, steps_per_pass=c["spp"])
        return dict(c=c, s=e, phi=torch.cat([f.reshape(-1) for f in fields]))
    if kind == "adjoint":
        phi, K, u, target = _adjoint_inputs(c, seed)
        return dict(c=c, leaves=[t.requires_grad_(True) for t in (phi, K, u)], target=target)
    d = _grid3_inputs(c, seed)
    s = Solver3(c["nx"], c["ny"], c["nz"], prec=c["prec"], bc=(c["bcx"], c["bcy"], c["bcz"]), phi_wall=d["walls"])
    s.set_coeffs(conv=c["conv"], u=U3[c["conv"]], diff=c["diff"], K=K3, se=SE3, r1=c["r1"])
    return dict(c=c, s=s, phi=d["phi"])


def run(state):
    c = state["c"]
    if c["kind"] == "adjoint":
        from paper_1603_09577_gb300 import adjoint
        phi, K, u = state["leaves"]
        out = adjoint.run(phi, K, u, c["steps"], ckpt_every=c["every"], prec=c["prec"], s_rates=RATES)
        loss = 0.5 * ((out - state["target"]) ** 2).sum()
        grads = torch.autograd.grad(loss, (phi, K, u))
        return {"phi": out.detach().to(_real(c["prec"])), "dphi0": grads[0], "dK": grads[1], "du": grads[2]}
    s = state["s"]
    s.set_phi(state["phi"])
    s.step(c["steps"])
    if c["kind"] == "ensemble":
        return {"phi": s.phi(torch.float32)}
    out = {"phi": s.phi(_real(c["prec"]))}
    if c.get("stats"):
        # the eight device-side statistics (sums, largest value, count of non-finite nodes)
        out["stats"] = s.reduce_async(out=torch.empty(8, dtype=torch.float64, device="cuda"))
    return out


# operations per node and step of the collision: moments, equilibrium, relaxation, back-transform
FLOPS2, FLOPS3, FLOPS_ADJ = 130, 220, 330


def work(case):
    c = case
    if c["kind"] == "grid3":
        n = c["nx"] * c["ny"] * c["nz"]
    elif c["kind"] == "ensemble":
        n = sum(m * m for m in _sides(c))
    elif c["kind"] == "general":
        n = c["n"] * c["n"]
    else:
        n = c["nx"] * c["ny"]
    b = 8 if c.get("prec") == "f64" else 4
    by = 2 * n * b                                    # phi0 in, phi out
    if c["kind"] == "adjoint":
        # phi0, K and the target in, phi and the gradients out
        return {"bytes": (1 + 3 + 1 + 1 + 1 + 3) * n * b, "flops": float(n) * c["steps"] * (FLOPS2 + FLOPS_ADJ)}
    if c["kind"] == "grid" and c["cellk"]:
        by += 3 * n * 8
    if c["kind"] == "general":
        by += 4 * c["n"] * 8 * c["steps"]             # the wall values of every step
    return {"bytes": by, "flops": float(n) * c["steps"] * (FLOPS3 if c["kind"] == "grid3" else FLOPS2)}


# ---- the same jobs in 64 bits ------------------------------------------------------

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W2 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _moment_matrix():
    """Rows rho, e, eps, jx, qx, jy, qy, pxx, pxy over the nine velocities."""
    x, y = np.array(CX, float), np.array(CY, float)
    q = x * x + y * y
    return np.stack([np.ones(9), 3 * q - 4, 4 - 10.5 * q + 4.5 * q * q, x, (3 * q - 5) * x, y, (3 * q - 5) * y,
                     x * x - y * y, x * y])


class _Lattice2:
    """D2Q9 MRT in FP64 torch operations, Scheme B with R = r1 phi or (a) Scheme A with R = b phi (1 - phi).
    K: three numbers, or a field (3, ny, nx)."""

    def __init__(self, phi0, conv, u, diff, K, s, r1=0.0, abb=(False, False), walls=(0.0,) * 4, a=False, b=0.0):
        self.conv, self.u, self.diff, self.s, self.r1 = conv, u, diff, s, r1
        self.abb, self.walls, self.a, self.b = abb, walls, a, b
        dev = phi0.device
        M = _moment_matrix()
        self.M = torch.tensor(M, device=dev)
        self.Mi = torch.tensor(np.linalg.inv(M), device=dev)
        ka, kb, kc = 3.0 * K[0] + 0.5, 3.0 * K[1], 3.0 * K[2] + 0.5
        det = ka * kc - kb * kb
        self.A = (kc / det, -kb / det, ka / det)
        self.ny, self.nx = phi0.shape
        self.f = self.start(phi0)
        self.phi_prev = phi0
        self.f = self.collide(self.f, phi0)
        self.links = self.wall_links()

    def coef(self, phi):
        ux, uy = self.u
        if self.conv == 0:
            B, Bp, C = (ux * phi, uy * phi), (ux, uy), phi
        else:
            B, Bp, C = (ux * phi * phi / 2, uy * phi * phi / 2), (ux * phi, uy * phi), phi ** 3 / 3
        g = phi if self.diff == 0 else phi + phi ** 2 / 2 if self.diff == 1 else phi + phi ** 3 / 3
        return B, Bp, (ux * ux * C + g / 3, ux * uy * C, uy * uy * C + g / 3)

    def feq(self, phi):
        B, _, (cxx, cxy, cyy) = self.coef(phi)
        qxx, qyy = cxx - phi / 3, cyy - phi / 3
        return torch.stack([W2[k] * (phi + 3 * (CX[k] * B[0] + CY[k] * B[1]) +
                                     4.5 * (qxx * (CX[k] ** 2 - 1 / 3) + 2 * CX[k] * CY[k] * cxy + qyy * (CY[k] ** 2 - 1 / 3)))
                            for k in range(9)])

    def start(self, phi):
        f = self.feq(phi)
        if not self.a and self.r1:
            _, Bp, _ = self.coef(phi)
            R = self.r1 * phi
            f = f - 0.5 * torch.stack([W2[k] * (1 + 3 * (CX[k] * Bp[0] + CY[k] * Bp[1])) * R for k in range(9)])
        return f

    def wall_links(self):
        """(crossed walls, k, rows, columns, feq_k + feq_opp(k) at the wall value) of the links whose
        source lies beyond a wall; those that cross two walls, at the corners, come last."""
        rows = [(slice(None), None)] + [(slice(0, 1), 2), (slice(self.ny - 1, self.ny), 3)] * self.abb[1]
        cols = [(slice(None), None)] + [(slice(0, 1), 0), (slice(self.nx - 1, self.nx), 1)] * self.abb[0]
        links = []
        for k in range(1, 9):
            for sy, wy in rows:
                for sx, wx in cols:
                    if (wy is not None and CY[k] != (1 if wy == 2 else -1)) or (wx is not None and CX[k] != (1 if wx == 0 else -1)):
                        continue
                    vals = [self.walls[w] for w in (wx, wy) if w is not None]
                    if vals:
                        e = self.feq(torch.tensor(sum(vals) / len(vals), dtype=torch.float64, device=self.f.device))
                        links.append((len(vals), k, sy, sx, e[k] + e[OPP[k]]))
        return sorted(links, key=lambda t: t[0])

    def pull(self):
        f = torch.stack([torch.roll(self.f[k], (CY[k], CX[k]), (0, 1)) for k in range(9)])
        for _, k, sy, sx, v in self.links:
            f[k][sy, sx] = v - self.f[OPP[k]][sy, sx]
        return f

    def nee(self, f, rec):
        """Extrapolated Dirichlet nodes on all four sides: feq(phi_b) plus the inward neighbour's rest."""
        n = self.nx
        rest = f - self.feq(f.sum(0))
        idx = torch.arange(n, device=f.device).clamp(1, n - 2)
        out = f.clone()
        west, east, south, north = rec[:n], rec[n:2 * n], rec[2 * n:3 * n], rec[3 * n:]
        out[:, 0, :] = self.feq(south) + rest[:, 1, :][:, idx]
        out[:, -1, :] = self.feq(north) + rest[:, -2, :][:, idx]
        out[:, :, 0] = self.feq(west) + rest[:, :, 1][:, idx]
        out[:, :, -1] = self.feq(east) + rest[:, :, -2][:, idx]
        return out

    def collide(self, f, prev=None):
        s = self.s
        m = (self.M @ f.reshape(9, -1)).reshape(f.shape)
        rho = m[0]
        phi = rho if self.a else rho / (1 - 0.5 * self.r1)
        B, Bp, (cxx, cxy, cyy) = self.coef(phi)
        A3, A35, A5 = self.A
        d3, d5 = m[3] - B[0], m[5] - B[1]
        dm = [torch.zeros_like(rho), -s[1] * (m[1] - (3 * (cxx + cyy) - 4 * phi)), -s[2] * (m[2] - 3 * (phi - cxx - cyy)),
              -(A3 * d3 + A35 * d5), -s[4] * (m[4] + B[0]), -(A35 * d3 + A5 * d5), -s[6] * (m[6] + B[1]),
              -s[7] * (m[7] - (cxx - cyy)), -s[8] * (m[8] - cxy)]
        if self.a:
            _, Bq, _ = self.coef(prev)
            R1, R0 = self.b * phi * (1 - phi), self.b * prev * (1 - prev)
            t = lambda q: (q[0] - 0.5 * (A3 * q[0] + A35 * q[1]), q[1] - 0.5 * (A35 * q[0] + A5 * q[1]))  # noqa: E731
            t1, t0 = t(Bp), t(Bq)
            R = 1.5 * R1 - 0.5 * R0
            Sx, Sy = 1.5 * t1[0] * R1 - 0.5 * t0[0] * R0, 1.5 * t1[1] * R1 - 0.5 * t0[1] * R0
            for j, v in ((0, R), (1, -2 * R), (2, R), (3, Sx), (4, -Sx), (5, Sy), (6, -Sy)):
                dm[j] = dm[j] + v
            self.phi_prev = phi
        elif self.r1:
            R = self.r1 * phi
            sx, sy = Bp[0] * R, Bp[1] * R
            for j, v in ((0, R), (1, -2 * (1 - s[1] / 2) * R), (2, (1 - s[2] / 2) * R),
                         (3, sx - 0.5 * (A3 * sx + A35 * sy)), (4, -(1 - s[4] / 2) * sx),
                         (5, sy - 0.5 * (A35 * sx + A5 * sy)), (6, -(1 - s[6] / 2) * sy)):
                dm[j] = dm[j] + v
        return f + (self.Mi @ torch.stack(dm).reshape(9, -1)).reshape(f.shape)

    def steps(self, n, rec=None):
        for i in range(n):
            f = self.pull()
            if rec is not None:
                f = self.nee(f, rec[i])
            self.f = self.collide(f, self.phi_prev)
        return self

    def phi(self):
        return self.phi_prev if self.a else self.f.sum(0) / (1 + 0.5 * self.r1)


def _exact_grid(c, seed):
    d = _grid_inputs(c, seed)
    K = d["K"] if c["cellk"] else (c["kxx"], c["kxy"], c["kyy"])
    L = _Lattice2(d["phi"].double(), c["conv"], (c["ux"], c["uy"]), c["diff"], K, RATES, c["r1"],
                  (c["bcx"] == "abb", c["bcy"] == "abb"), d["walls"])
    phi = L.steps(c["steps"]).phi()
    out = {"phi": phi}
    if c.get("stats"):
        z = torch.zeros((), dtype=torch.float64, device=phi.device)
        out["stats"] = torch.stack([phi.sum(), z, z, z, z, phi.abs().max(), z, (phi * phi).sum()])
    return out


def _exact_adjoint(c, seed):
    phi0, K, u, target = (t.double() for t in _adjoint_inputs(c, seed))

    def start(phi, K, u):
        return _Lattice2(phi, 0, (u[0], u[1]), 0, K, RATES)

    with torch.no_grad():
        L = start(phi0, K, u)
        states = [L.f]
        for _ in range(c["steps"]):
            L.f = L.collide(L.pull())
            states.append(L.f)
    out = states.pop().sum(0)
    lam = (out - target).expand(9, -1, -1)
    gK, gu = torch.zeros_like(K), torch.zeros_like(u)
    for F in reversed(states):
        F, k, v = F.clone().requires_grad_(True), K.clone().requires_grad_(True), u.clone().requires_grad_(True)
        L = start(phi0, k, v)
        L.f = F
        lam, a, b = torch.autograd.grad(L.collide(L.pull()), (F, k, v), lam)
        gK += a
        gu += b
    p, k, v = phi0.clone().requires_grad_(True), K.clone().requires_grad_(True), u.clone().requires_grad_(True)
    dphi, a, b = torch.autograd.grad(start(p, k, v).f, (p, k, v), lam)
    # the initial collision acts on an equilibrium and leaves it as it is: no gradient in K there
    return {"phi": out, "dphi0": dphi, "dK": gK + a, "du": gu + b}


CX3 = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, -1, 1, 0, 0, 0, 0)
CY3 = (0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1)
CZ3 = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, -1, 1)


def _exact_grid3(c, seed):
    d = _grid3_inputs(c, seed)
    phi0, u, r1, walls = d["phi"].double(), U3[c["conv"]], c["r1"], d["walls"]
    Km = np.array([[K3[0], K3[1], K3[2]], [K3[1], K3[3], K3[4]], [K3[2], K3[4], K3[5]]])
    G = np.linalg.inv(3 * Km + 0.5 * np.eye(3)) - SE3 * np.eye(3)
    cs = list(zip(CX3, CY3, CZ3))
    w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    opp = [0] + [k + 1 if k % 2 else k - 1 for k in range(1, 19)]
    u2 = sum(v * v for v in u)

    def parts(phi):
        beta, bp, C = (phi, 1.0, phi) if c["conv"] == 0 else (phi * phi / 2, phi, phi ** 3 / 3)
        iso = 0 * phi if c["diff"] == 0 else phi * phi / 6 if c["diff"] == 1 else phi ** 3 / 9
        return beta, bp, C, iso

    def feq(k, phi, q):
        beta, _, C, iso = q
        cu, c2 = sum(a * b for a, b in zip(cs[k], u)), sum(a * a for a in cs[k])
        return w[k] * (phi + 3 * cu * beta + 4.5 * ((cu * cu - u2 / 3) * C + (c2 - 1) * iso))

    def collide(f):
        phi = sum(f) / (1 - 0.5 * r1)
        q = parts(phi)
        beta, bp, _, _ = q
        R = r1 * phi
        v = [sum(cs[k][a] * f[k] for k in range(19) if cs[k][a]) - u[a] * (beta - bp * R / 2) for a in range(3)]
        g = [sum(G[a, b] * v[b] for b in range(3)) / 10 for a in range(3)]
        out = []
        for k in range(19):
            cu = sum(a * b for a, b in zip(cs[k], u))
            x = f[k] - SE3 * (f[k] - feq(k, phi, q)) + (1 - SE3 / 2) * w[k] * (1 + 3 * cu * bp) * R
            for a in range(3):
                if cs[k][a]:
                    x = x - cs[k][a] * g[a]
            out.append(x)
        return out

    abb = [c["bcx"] == "abb", c["bcy"] == "abb", c["bcz"] == "abb"]
    dims = (c["nx"], c["ny"], c["nz"])
    beyond = []                                       # (k, slices, value): links that cross one or more walls
    for k in range(1, 19):
        sides = [[(slice(None), None)] for _ in range(3)]
        for a in range(3):
            if abb[a] and cs[k][a]:
                at = 0 if cs[k][a] > 0 else dims[a] - 1
                sides[a].append((slice(at, at + 1), walls[2 * a + (0 if cs[k][a] > 0 else 1)]))
        for sx in sides[0]:
            for sy in sides[1]:
                for sz in sides[2]:
                    vals = [t[1] for t in (sx, sy, sz) if t[1] is not None]
                    if vals:
                        p = torch.tensor(sum(vals) / len(vals), dtype=torch.float64, device=phi0.device)
                        q = parts(p)
                        beyond.append((len(vals), k, (sz[0], sy[0], sx[0]), feq(k, p, q) + feq(opp[k], p, q)))
    beyond.sort(key=lambda t: t[0])
    q0 = parts(phi0)
    f = [feq(k, phi0, q0) - 0.5 * w[k] * (1 + 3 * sum(a * b for a, b in zip(cs[k], u)) * q0[1]) * r1 * phi0 for k in range(19)]
    f = collide(f)
    for _ in range(c["steps"]):
        g = [torch.roll(f[k], (cs[k][2], cs[k][1], cs[k][0]), (0, 1, 2)) for k in range(19)]
        for _, k, at, v in beyond:
            g[k][at] = v - f[opp[k]][at]
        f = collide(g)
    return {"phi": sum(f) / (1 + 0.5 * r1)}


def exact(case, seed):
    c = case
    if c["kind"] == "grid":
        return _exact_grid(c, seed)
    if c["kind"] == "general":
        d = _fisher_inputs(c, seed)
        # delta = 1: the power-law flux is the quadratic one
        L = _Lattice2(d["phi"].double(), 1, (d["ax"], 0.0), 0, (d["K"], 0.0, d["K"]), RATES, a=True, b=d["b"])
        return {"phi": L.steps(c["steps"], d["rec"]).phi()}
    if c["kind"] == "ensemble":
        inst, fields = _ensemble_inputs(c, seed)
        return {"phi": torch.cat([_Lattice2(f.double(), 0, i["u"], 1, i["K"], i["s"]).steps(c["steps"]).phi().reshape(-1)
                                  for i, f in zip(inst, fields)])}
    if c["kind"] == "adjoint":
        return _exact_adjoint(c, seed)
    return _exact_grid3(c, seed)
