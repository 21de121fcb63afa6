"""The workloads of this library that are timed, and their values in 64 bits.

Every case is one output interval as a user's program runs it through the
public binding: the initial field goes in, the solver advances it, the field
(and the state, or the gradients) comes out.  The solver object, its mesh and
its coefficients are what such a program keeps between intervals.

``exact`` restates the method in plain torch float64 on one list of velocity
planes (arXiv:1906.11036, the step summary of Section 2), in any number of
dimensions, with autograd for the gradients; it shares no code with the
library.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1906_11036_gb300 import inputs as I
from paper_1906_11036_gb300.dugks import BatchSolver, Solver, Solver3

PER, DIR = I.PERIODIC, I.DIRICHLET


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the linear Gaussian hill in double precision, host arrays in and out: the smallest call a
        # user makes, where every step is a few microseconds of work
        dict(name="hill_64_fp64_host", kind="step", form="hill", nx=64, ny=64, prec=64, steps=200, host=True),
        # Example 4.4 (full diffusion tensor) on the paper's own 400^2 grid, double precision
        dict(name="aniso_400_fp64", kind="step", form="aniso", nx=400, ny=400, prec=64, steps=50, host=False),
        # a small ragged grid in single precision: launches and latency
        dict(name="burgers_70x45_fp32", kind="step", form="burgers", nx=70, ny=45, prec=32, steps=200, host=False),
        # a mid-sized ragged grid with walls on both axes of a stretched mesh
        dict(name="mixed_330x517_fp32", kind="step", form="mixed", nx=330, ny=517, prec=32, steps=100, host=False),
        # the nonlinear Burgers-type workload: both state buffers fit in L2
        dict(name="burgers_1024_fp32", kind="step", form="burgers", nx=1024, ny=1024, prec=32, steps=100, host=False),
        # nonlinear diffusion on the stretched mesh with walls: the state does not fit in L2
        dict(name="nonuniform_2048_fp32", kind="step", form="nonuniform", nx=2048, ny=2048, prec=32, steps=50, host=False),
        # Example 4.1 with its source term, on a grid of the paper's size
        dict(name="cde_source_200_fp32", kind="source", form="cde", nx=200, ny=200, prec=32, steps=100),
        # Example 4.5: six source terms and a tensor D, on a large grid
        dict(name="nonlinear_source_2048_fp32", kind="source", form="nonlinear", nx=2048, ny=2048, prec=32, steps=20),
        # the gradient workload: periodic Burgers-type NCDE, a checkpoint every 20 steps
        dict(name="gradient_512_fp32", kind="gradient", form="burgers", nx=512, ny=512, prec=32, steps=40, every=20, with_u=False),
        # the gradient on the large stretched mesh with walls, the velocity's derivative with it
        dict(name="gradient_walls_2048_fp32", kind="gradient", form="nonuniform", nx=2048, ny=2048, prec=32, steps=10, every=5, with_u=True),
        # 256 independent instances of sides 64 .. 512 advanced together
        dict(name="batch_256_fp32", kind="batch", count=256, smallest=64, largest=512, odd=False, steps=100),
        # the three-dimensional Burgers-type workload
        dict(name="d3q19_256_fp32", kind="step3", form="burgers", nx=256, ny=256, nz=256, lattice=19, prec=32, steps=10),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["step", "step", "step", "step64", "step64", "source", "gradient", "batch", "step3", "step3"])
    if kind == "step":
        return dict(kind="step", form=rng.choice(["burgers", "nonuniform", "mixed", "hill"]), nx=log(40, 2048),
                    ny=log(40, 2048), prec=32, steps=rng.choice([20, 50, 100]), host=rng.random() < 0.2)
    if kind == "step64":
        return dict(kind="step", form=rng.choice(["hill", "aniso", "burgers", "nonuniform"]), nx=log(32, 512),
                    ny=log(32, 512), prec=64, steps=rng.choice([20, 50, 100]), host=rng.random() < 0.5)
    if kind == "source":
        form = rng.choice(["cde", "nonlinear"])
        n = log(64, 1024)  # the presets are square
        return dict(kind="source", form=form, nx=n, ny=n, prec=rng.choice([32, 32, 64]) if n <= 256 else 32,
                    steps=rng.choice([20, 50]))
    if kind == "gradient":
        return dict(kind="gradient", form=rng.choice(["burgers", "nonuniform"]), nx=log(48, 1024), ny=log(48, 1024),
                    prec=32, steps=rng.choice([12, 20, 30]), every=rng.choice([5, 10, 20]), with_u=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind="batch", count=log(4, 24), smallest=rng.choice([32, 64]), largest=rng.choice([128, 256]),
                    odd=True, steps=rng.choice([20, 50, 100]))
    prec = rng.choice([32, 32, 32, 64])
    top = 160 if prec == 32 else 64
    return dict(kind="step3", form=rng.choice(["burgers", "walls"]), nx=log(24, top), ny=log(24, top), nz=log(24, top),
                lattice=rng.choice([15, 19]), prec=prec, steps=rng.choice([5, 10]))


# ---------------------------------------------------------------------------
# problems and their initial fields (from the seed alone)
# ---------------------------------------------------------------------------

def _waves(xc, yc, kmax, seed):
    """Random plane waves |kx|, |ky| <= kmax of unit RMS on the grid [ny, nx] (float64, on the GPU)."""
    g = torch.Generator().manual_seed(int(seed) % (1 << 62))
    k = torch.arange(-kmax, kmax + 1, dtype=torch.float64)
    A, B = (torch.randn(len(k), len(k), dtype=torch.float64, generator=g).cuda() for _ in range(2))
    A[kmax, kmax] = B[kmax, kmax] = 0.0
    ax = 2 * math.pi * torch.outer(torch.as_tensor(xc), k).cuda()
    ay = 2 * math.pi * torch.outer(torch.as_tensor(yc), k).cuda()
    cx, sx, cy, sy = ax.cos(), ax.sin(), ay.cos(), ay.sin()
    v = cy @ A @ cx.T - sy @ A @ sx.T + cy @ B @ sx.T + sy @ B @ cx.T
    return v / v.square().mean().sqrt()


def _grid(xc, yc):
    return torch.as_tensor(xc).cuda()[None, :], torch.as_tensor(yc).cuda()[:, None]


def _problem(case, seed):
    """(problem, phi0 float64 on the GPU) of a 2-D case."""
    nx, ny, form = case["nx"], case["ny"], case["form"]
    if case["kind"] == "source":
        p, _ = (I.cde_source if form == "cde" else I.nonlinear_source)(nx)
        xc, yc = p.centres()
        X, Y = _grid(xc, yc)
        if form == "cde":
            base = (math.pi * (X + Y)).sin()
            return p, base + 0.02 * _waves(xc / 2, yc / 2, 3, seed)
        return p, 1.1 - (2 * math.pi * X).cos() * (2 * math.pi * Y).cos() + 0.02 * _waves(xc, yc, 3, seed)
    if form == "hill":
        xf, yf = I.uniform_faces(nx, 0.0, 2.0), I.uniform_faces(ny, 0.0, 2.0)
        p = I.Problem(xf=xf, yf=yf, c=1.0, u=(0.1, 0.1), b=(0.0, 1.0), alpha=0.01, d=(0.0, 1.0),
                      dt=I.cfl_dt(xf, yf, 1.0, 0.5))
    elif form == "aniso":
        xf, yf = I.uniform_faces(nx, -1.0, 1.0), I.uniform_faces(ny, -1.0, 1.0)
        p = I.Problem(xf=xf, yf=yf, c=1.0, u=(0.01, 0.01), b=(0.0, 1.0), alpha=1e-3, d=(0.0,),
                      d_tensor=((0.0, 1.0), (0.0, 1.0), (0.0, 2.0)), dt=I.cfl_dt(xf, yf, 1.0, 0.5))
    elif form == "burgers":
        xf, yf = I.uniform_faces(nx), I.uniform_faces(ny)
        p = I.Problem(xf=xf, yf=yf, c=10.0, u=(1.0, 1.0), b=(0.0, 0.0, 0.5), alpha=0.005, d=(0.0, 1.0),
                      dt=I.cfl_dt(xf, yf, 10.0, 0.4))
    elif form == "nonuniform":
        xf, yf = I.tanh_faces(nx, 2.0), I.tanh_faces(ny, 2.0)
        p = I.Problem(xf=xf, yf=yf, bc=(DIR,) * 4, bc_value=(1.0, 0.5, 0.5, 0.5), c=10.0, u=(0.05, 0.0),
                      b=(0.0, 1.0), alpha=0.01, d=(0.0, 0.0, 1.0), dt=I.cfl_dt(xf, yf, 10.0, 0.4))
    else:  # "mixed": stretched walls in x and y, quadratic B, quadratic D
        xf, yf = I.tanh_faces(nx, 1.5), I.tanh_faces(ny, 1.5)
        p = I.Problem(xf=xf, yf=yf, bc=(DIR,) * 4, bc_value=(1.2, 0.6, 0.9, 0.7), c=10.0, u=(0.3, -0.2),
                      b=(0.0, 0.0, 0.5), alpha=0.02, d=(0.0, 1.0, 0.5), dt=I.cfl_dt(xf, yf, 10.0, 0.45))
    xc, yc = p.centres()
    X, Y = _grid(xc, yc)
    if form in ("hill", "aniso"):
        x0 = 1.0 if form == "hill" else 0.0
        w = _waves(xc / 2, yc / 2, 2, seed)
        return p, torch.exp(-((X - x0) ** 2 + (Y - x0) ** 2) / 0.02) * (1 + 0.05 * torch.tanh(w)) + 0.01
    if form == "burgers":
        return p, 1 + 0.2 * (2 * math.pi * X).sin() * (2 * math.pi * Y).sin() + 0.01 * _waves(xc, yc, 8, seed)
    return p, 1 + 0.5 * torch.tanh(_waves(xc, yc, 2, seed))


def _problem3(case, seed):
    """(problem, phi0 float64 [nz, ny, nx] on the GPU) of a 3-D case."""
    n = (case["nx"], case["ny"], case["nz"])
    if case["form"] == "burgers":
        f = [I.uniform_faces(m) for m in n]
        p = I.Problem3(xf=f[0], yf=f[1], zf=f[2], lattice=case["lattice"], c=10.0, u=(1.0, 1.0, 1.0), b=(0.0, 0.0, 0.5),
                       alpha=0.005, d=(0.0, 1.0), dt=I.cfl_dt3(*f, 10.0, 0.4))
    else:
        f = [I.tanh_faces(m, 1.4) for m in n]
        p = I.Problem3(xf=f[0], yf=f[1], zf=f[2], bc=(DIR,) * 6, bc_value=(1.2, 0.6, 0.9, 0.7, 1.1, 0.8),
                       lattice=case["lattice"], c=4.0, u=(0.3, -0.2, 0.15), b=(0.0, 1.0), alpha=0.02, d=(0.0, 0.0, 1.0),
                       dt=I.cfl_dt3(*f, 4.0, 0.4))
    x, y, z = (torch.as_tensor(a).cuda() for a in p.centres())
    X, Y, Z = x[None, None, :], y[None, :, None], z[:, None, None]
    g = np.random.default_rng(seed)
    v = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
    for _ in range(8):
        k = 2 * math.pi * g.integers(-4, 5, size=3)
        v += g.standard_normal() * torch.cos(k[0] * X + k[1] * Y + k[2] * Z + g.uniform(0, 2 * math.pi))
    tp = 2 * math.pi
    return p, 1 + 0.2 * (tp * X).sin() * (tp * Y).sin() * (tp * Z).sin() + 0.01 * v


def _batch(case, seed):
    """The instances (side, a, D0, phi0 seed) of a batched case; coefficients and fields from the seed."""
    g = np.random.default_rng(seed)
    if case["odd"]:
        sides = np.round(np.geomspace(case["smallest"], case["largest"], case["count"]))
    else:
        steps = int(math.log2(case["largest"] // case["smallest"])) + 1
        sides = np.resize([case["smallest"] << k for k in range(steps)], case["count"])
    sides = g.permutation(sides)  # the sizes are the case's, their order the seed's
    a, d0 = g.uniform(0.5, 2.0, case["count"]), g.uniform(0.002, 0.02, case["count"])
    items = []
    for i in range(case["count"]):
        xf = I.uniform_faces(int(sides[i]))
        p = I.Problem(xf=xf, yf=xf.copy(), c=10.0, u=(1.0, 1.0), b=(0.0, 0.0, 0.5 * float(a[i])), alpha=float(d0[i]),
                      d=(1.0, 0.0, 1.0), dt=I.cfl_dt(xf, xf, 10.0, 0.4))
        xc, yc = p.centres()
        X, Y = _grid(xc, yc)
        phi0 = 1 + 0.2 * (2 * math.pi * X).sin() * (2 * math.pi * Y).sin() + 0.01 * _waves(xc, yc, 8, seed + 1 + i)
        items.append((p, phi0.float()))
    return items


def _dtype(case):
    return torch.float64 if case.get("prec") == 64 else torch.float32


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        items = _batch(case, seed)
        return dict(case=case, solver=BatchSolver([p for p, _ in items]), phi0=[f for _, f in items])
    if kind == "step3":
        p, phi0 = _problem3(case, seed)
        return dict(case=case, solver=Solver3(p, precision=case["prec"]), phi0=phi0.to(_dtype(case)))
    p, phi0 = _problem(case, seed)
    s = dict(case=case, solver=Solver(p, precision=case["prec"]), phi0=phi0.to(_dtype(case)))
    if case.get("host"):
        s["phi0"] = s["phi0"].double().cpu().numpy()
    if kind == "gradient":
        s["misfit"] = _misfit(p, phi0, seed).to(_dtype(case))
    return s


def _misfit(p, phi0, seed):
    """dJ/dphi^N of a field misfit: the cell areas (scaled to order one) times the distance from a smooth target."""
    area = torch.as_tensor(np.outer(np.diff(p.yf), np.diff(p.xf))).cuda()
    return area / area.mean() * (phi0 - 1 - 0.02 * _waves(*p.centres(), 4, seed + 77))


def run(state):
    case, s = state["case"], state["solver"]
    kind = case["kind"]
    if kind == "gradient":
        out = s.gradient(state["phi0"], case["steps"], state["misfit"], checkpoint_every=case["every"],
                         with_u=case["with_u"])
        # the parameter gradients are sums of single-precision terms
        got = {"phi0": out[0], "alpha": np.float32(out[1])}
        if case["with_u"]:
            got["u"] = np.array(out[2], dtype=np.float32)
        return got
    if kind == "batch":
        for i, f in enumerate(state["phi0"]):
            s.init_phi(i, f)
        s.step(case["steps"])
        got = {}
        for i, f in enumerate(state["phi0"]):  # the fields, by the side of their grids
            got.setdefault(_group(f.shape[0]), []).append(s.get_phi(i).reshape(-1))
        s.sync()
        return {k: torch.cat(v) for k, v in got.items()}
    s.init_phi(state["phi0"])
    s.step(case["steps"])
    if case.get("host"):
        phi, mass = s.get_phi_host()
        return {"phi": phi.astype(np.float32) if case["prec"] == 32 else phi, "mass": np.float32(mass)}
    return {"phi": s.get_phi(), "f": s.save_state()}


def _group(side):
    return "to_%d" % (64 << max(0, math.ceil(math.log2(side / 64))))


def work(case):
    """ftilde read once and written once per step (and per adjoint step also mu read and lambda written); the
    operations are those of the step's formulas per velocity: equilibrium, transforms, the faces and the update."""
    q = case.get("lattice", 9)
    size = 8 if case.get("prec") == 64 else 4
    if case["kind"] == "batch":
        s0, s1, n = case["smallest"], case["largest"], case["count"]
        if case["odd"]:  # the mean of side^2 for sides spread evenly over the logarithm
            cells = n * (s1 * s1 - s0 * s0) / (2 * math.log(s1 / s0))
        else:
            k = int(math.log2(s1 // s0)) + 1
            cells = n * sum((s0 << i) ** 2 for i in range(k)) / k
    else:
        cells = case["nx"] * case["ny"] * case.get("nz", 1)
    per_step = 2 * q * size
    flops = (40 if case["kind"] != "step3" else 60) * q
    if case["kind"] == "source":
        per_step += size * ((1 if case["form"] == "cde" else 6) + 2)
        flops += 60
    steps = case["steps"]
    if case["kind"] == "gradient":  # forward, and the reverse sweep, which reads the state and mu and writes lambda
        return {"bytes": cells * steps * (per_step + 3 * q * size), "flops": cells * steps * flops * 3.0}
    return {"bytes": cells * (steps * per_step + 2 * size), "flops": cells * steps * float(flops)}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------

_D2Q9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_D3Q19 = [(0, 0, 0)] + [tuple(s * (a == b) for b in range(3)) for a in range(3) for s in (1, -1)] + [
    (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (-1, 0, 1), (1, 0, -1),
    (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_D3Q15 = _D3Q19[:7] + [(1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1), (-1, -1, -1), (-1, -1, 1), (-1, 1, -1), (1, -1, -1)]
_WEIGHTS = {9: (4 / 9, 1 / 9, 1 / 36, 0), 19: (1 / 3, 1 / 18, 1 / 36, 0), 15: (2 / 9, 1 / 9, 0, 1 / 72)}


def _poly(coef, x):
    v = torch.zeros_like(x) + coef[-1]
    for a in reversed(coef[:-1]):
        v = v * x + a
    return v


class _Method:
    """One DUGKS step on a list of velocity planes (trailing dimensions [z,] y, x)."""

    def __init__(self, faces, bc, bcv, q, c, u, b, alpha, d, dt, tensor=None, source=(), t0=0.0):
        self.e = {9: _D2Q9, 15: _D3Q15, 19: _D3Q19}[q]
        self.w = [_WEIGHTS[q][sum(map(abs, e))] for e in self.e]
        self.dim, self.c, self.u, self.b, self.d, self.dt, self.tensor = len(faces), c, u, list(b), list(d), dt, tensor
        # int_0^phi b'^2 as polynomial coefficients (Remark 3)
        self.ci = [0.0] * max(2, 2 * len(self.b))
        for k in range(1, len(self.b)):
            for m in range(1, len(self.b)):
                self.ci[k + m - 1] = self.ci[k + m - 1] + k * m * self.b[k] * self.b[m] / (k + m - 1)
        self.bc, self.bcv = bc, bcv
        self.h = 0.5 * dt
        lam = self.lam = alpha * 3.0 / (c * c)
        self.abp, self.bbp = (2 * lam - self.h) / (2 * lam + dt), 3 * self.h / (2 * lam + dt)
        self.atp, self.btp = (2 * lam - dt) / (2 * lam + dt), 2 * dt / (2 * lam + dt)
        self.af, self.bf = 2 * lam / (2 * lam + self.h), self.h / (2 * lam + self.h)
        self.axes = [self._axis(np.asarray(f, dtype=np.float64), bc[2 * a] == PER, a) for a, f in enumerate(faces)]
        self.source, self.t, self.before = source, t0, None

    def _axis(self, f, per, a):
        n = len(f) - 1
        x = np.empty(n + 2)
        x[1:-1] = 0.5 * (f[1:] + f[:-1])
        x[0], x[-1] = (x[n] - (f[n] - f[0]), x[1] + (f[n] - f[0])) if per else (2 * f[0] - x[1], 2 * f[n] - x[n])
        gap = np.diff(x)
        w = (f - x[:-1]) / gap
        tl, tr = 1 - w, w.copy()
        if not per:
            tl[0], tr[0], tl[-1], tr[-1] = 0, 1, 1, 0
        shape = [-1] + [1] * a
        t = lambda v: torch.as_tensor(v).cuda().reshape(shape)  # noqa: E731
        return dict(w=t(w), hcd=t(self.h * self.c / gap), tl=t(self.h * self.c * tl), tr=t(self.h * self.c * tr),
                    ig=t(1 / (x[2:] - x[:-2])), r=t(self.dt * self.c / np.diff(f)))

    def feq(self, phi):
        """Eq. 2.3 for every velocity."""
        b, ci, c = _poly(self.b, phi), _poly(self.ci, phi), self.c
        u2 = sum(v * v for v in self.u)
        if self.tensor is None:
            d = _poly(self.d, phi) - phi
        else:
            dxx, dxy, dyy = (_poly(list(v), phi) for v in self.tensor)
        out = []
        for e, w in zip(self.e, self.w):
            eu, e2 = sum(k * v for k, v in zip(e, self.u)), sum(k * k for k in e)
            if self.tensor is None:
                dd = (3 * e2 - self.dim) / 2 * d
            else:
                dd = (3 * e[0] ** 2 - 1) / 2 * dxx + 3 * e[0] * e[1] * dxy + (3 * e[1] ** 2 - 1) / 2 * dyy - (3 * e2 - 2) / 2 * phi
            out.append(w * (phi + 3 * eu / c * b + dd + (9 * eu * eu - 3 * u2) / (2 * c * c) * ci))
        return out

    def _pad(self, P, phi, a):
        """P (a list) with one more cell on both sides along axis a: (all low halves, all high halves)."""
        dim, n = -1 - a, P[0].shape[-1 - a]
        if self.bc[2 * a] == PER:
            lo, hi = [p.narrow(dim, n - 1, 1) for p in P], [p.narrow(dim, 0, 1) for p in P]
        else:
            lo, hi = [], []
            for side, at, to in ((0, 0, lo), (1, n - 1, hi)):  # the mirrored cell, its non-equilibrium part kept
                edge = phi.narrow(dim, at, 1)
                new, old = self.feq(2 * self.bcv[2 * a + side] - edge), self.feq(edge)
                to += [p.narrow(dim, at, 1) + x - y for p, x, y in zip(P, new, old)]
        return [torch.cat((l, p, r), dim) for l, p, r in zip(lo, P, hi)]

    def _sources(self, phi, P, U):
        def S(t, x):
            F = sum(math.exp(k.rate * t) * (x ** k.power) * f for k, f in self.source)
            return F, F * _poly([m * self.b[m] for m in range(1, len(self.b))], x)

        F, G = S(self.t, phi)
        Fo, Go = (F, G) if self.before is None else S(self.t - self.dt, self.before)
        cs2, h, wr = self.c ** 2 / 3, self.h, 2 * self.lam * self.h / (2 * self.lam + self.h)
        for i, (e, w) in enumerate(zip(self.e, self.w)):
            cu = self.c * sum(k * v for k, v in zip(e, self.u)) / cs2
            P[i] = P[i] + w * (wr * cu * (G + (G - Go) / 4) + h * (F + (F - Fo) / 4))
            U[i] = U[i] + w * self.dt * (cu * (1.5 * G - 0.5 * Go) + 1.5 * F - 0.5 * Fo)
        self.before, self.t = phi, self.t + self.dt

    def step(self, f):
        phi = sum(f)
        eq = self.feq(phi)
        P = [self.abp * x + self.bbp * y for x, y in zip(f, eq)]
        U = [self.atp * x + self.btp * y for x, y in zip(f, eq)]
        del eq
        if self.source:
            self._sources(phi, P, U)
        pads = [self._pad(P, phi, a) for a in range(self.dim)]
        for a, m in enumerate(self.axes):
            dim, n = -1 - a, P[0].shape[-1 - a]
            fb = []
            for i, e in enumerate(self.e):
                p = pads[a][i]
                v = (1 - m["w"] + e[a] * m["hcd"]) * p.narrow(dim, 0, n + 1) + (m["w"] - e[a] * m["hcd"]) * p.narrow(dim, 1, n + 1)
                for t in range(self.dim):
                    if t == a or e[t] == 0:
                        continue
                    o, k = pads[t][i], P[0].shape[-1 - t]
                    g = (o.narrow(-1 - t, 2, k) - o.narrow(-1 - t, 0, k)) * self.axes[t]["ig"]
                    per = self.bc[2 * a] == PER  # a wall's ghost has no slope of its own (its weight is zero)
                    lo, hi = (g.narrow(dim, n - 1, 1), g.narrow(dim, 0, 1)) if per else (torch.zeros_like(g.narrow(dim, 0, 1)),) * 2
                    v = v - e[t] * (m["tl"] * torch.cat((lo, g), dim) + m["tr"] * torch.cat((g, hi), dim))
                fb.append(v)
            eqb = self.feq(sum(fb))
            for i, e in enumerate(self.e):
                if e[a]:
                    x = self.af * fb[i] + self.bf * eqb[i]
                    U[i] = U[i] - e[a] * m["r"] * (x.narrow(dim, 1, n) - x.narrow(dim, 0, n))
        return U


def _method(p, alpha=None, u=None, source=()):
    return _Method([p.xf, p.yf], p.bc, p.bc_value, 9, p.c, p.u if u is None else u, p.b,
                   p.alpha if alpha is None else alpha, p.d, p.dt, p.d_tensor, source, p.t0)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "step3":
        p, phi0 = _problem3(case, seed)
        m = _Method([p.xf, p.yf, p.zf], p.bc, p.bc_value, p.lattice, p.c, p.u, p.b, p.alpha, p.d, p.dt)
        return _advance(m, phi0.to(_dtype(case)).double(), case["steps"])
    p, phi0 = _problem(case, seed)
    if kind == "gradient":
        return _exact_gradient(case, seed, p, phi0)
    phi0 = phi0.to(_dtype(case)).double()
    m = _method(p, source=[(k, torch.as_tensor(k.field).cuda()) for k in p.source])
    out = _advance(m, phi0, case["steps"])
    if case.get("host"):
        mass = (torch.as_tensor(np.outer(np.diff(p.yf), np.diff(p.xf))).cuda() * out["phi"]).sum()
        return {"phi": out["phi"].cpu().numpy(), "mass": mass}
    return out


def _advance(m, phi0, steps):
    with torch.no_grad():
        f = m.feq(phi0)
        for _ in range(steps):
            f = m.step(f)
        return {"phi": sum(f), "f": torch.stack(f)}


def _exact_gradient(case, seed, p, phi0_64):
    phi0 = phi0_64.to(_dtype(case)).double()
    g = _misfit(p, phi0_64, seed).to(_dtype(case)).double()
    leaf = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=True) for v in (p.alpha, *p.u)]
    phi0 = phi0.clone().requires_grad_(True)

    def step(*f):
        return tuple(_method(p, leaf[0], leaf[1:]).step(list(f)))

    f = tuple(_method(p, leaf[0], leaf[1:]).feq(phi0))
    for _ in range(case["steps"]):  # every step is computed again in the reverse sweep: one step's graph at a time
        f = torch.utils.checkpoint.checkpoint(step, *f, use_reentrant=False)
    (sum(f) * g).sum().backward()
    out = {"phi0": phi0.grad, "alpha": leaf[0].grad}
    if case["with_u"]:
        out["u"] = torch.stack((leaf[1].grad, leaf[2].grad))
    return out


def _exact_batch(case, seed):
    """Instances of one side together, up to 256 cells a side (the larger ones would take too long)."""
    items = _batch(case, seed)
    sides = {}
    for i, (p, _) in enumerate(items):
        sides.setdefault(p.nx, []).append(i)
    found = [None] * len(items)
    with torch.no_grad():
        for side, at in sides.items():
            if side > 256:
                continue
            col = lambda f: torch.tensor([f(items[i][0]) for i in at], dtype=torch.float64, device="cuda").reshape(-1, 1, 1)  # noqa: E731
            p = items[at[0]][0]
            m = _Method([p.xf, p.yf], p.bc, p.bc_value, 9, p.c, p.u, (0.0, 0.0, col(lambda q: q.b[2])), col(lambda q: q.alpha),
                        p.d, p.dt)
            phi = _advance(m, torch.stack([items[i][1] for i in at]).double(), case["steps"])["phi"]
            for k, i in enumerate(at):
                found[i] = phi[k].reshape(-1)
    got = {}
    for i, (p, _) in enumerate(items):
        got.setdefault(_group(p.nx), []).append(found[i])
    return {k: None if any(x is None for x in v) else torch.cat(v) for k, v in got.items()}
