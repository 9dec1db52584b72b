"""Workloads whose speed this package is measured by: what users of the solver
and of the warm-start network have them do, through the public Python binding.

Kinds of case:
  step      one grid: advance `steps` RK4 steps, then read every field (and, for
            the drop studies, the contact angle) back: a simulation between two
            of its output times
  sweep     a parameter sweep: `count` uneven 2D grids advanced together by one
            batched launch, then every field of every grid read back
  forward   one prediction of the network on device arrays
  train     one training step on host arrays, with loss and gradients

FP32-mixed fields are kept as float32 snapshots, the precision of that form's
state; FP64 fields as the doubles they are.
"""
import dataclasses
import math
import random

import numpy as np
import torch

from paper_2412_16843_gb300 import cdi, inputs

FP64, FP32 = "fp64", "fp32"


def listed():
    return [
        # the paper's equilibrium-drop study (mesh family of small 2D grids run for many steps,
        # angle and wetted length logged every chunk): the smallest grid, launch and barrier latency
        {"name": "drop2d_64x32_fp64", "kind": "step", "flow": "drop2d", "n": "64x32", "precision": FP64,
         "warm": "previous", "tol": 1e-12, "pre": 1, "post": 1, "cpre": -1, "cpost": -1, "steps": 10},
        # the paper's two-phase Couette flow in the parity precision, extrapolated first guesses
        {"name": "couette2d_512x128_fp64", "kind": "step", "flow": "couette2d", "n": "512x128", "precision": FP64,
         "warm": "extrapolated", "tol": 1e-12, "pre": 1, "post": 1, "cpre": -1, "cpost": -1, "steps": 4},
        # the same flow in the fast precision
        {"name": "couette2d_512x128_fp32", "kind": "step", "flow": "couette2d", "n": "512x128", "precision": FP32,
         "warm": "extrapolated", "tol": 1e-8, "pre": 1, "post": 1, "cpre": -1, "cpost": -1, "steps": 4},
        # 3D drop in the parity precision: the runs that generate the network's training pairs
        {"name": "drop3d_64_fp64", "kind": "step", "flow": "drop3d", "n": "64x64x64", "precision": FP64,
         "warm": "previous", "tol": 1e-12, "pre": 1, "post": 2, "cpre": -1, "cpost": -1, "steps": 2},
        # a 3D box that is no power of two and no multiple of the sweep's tiles
        {"name": "drop3d_224x96x96_fp32", "kind": "step", "flow": "drop3d", "n": "224x96x96", "precision": FP32,
         "warm": "previous", "tol": 1e-8, "pre": 1, "post": 2, "cpre": -1, "cpost": -1, "steps": 2},
        # the 256^3 drop with the library's default cycle
        {"name": "drop3d_256_fp32", "kind": "step", "flow": "drop3d", "n": "256x256x256", "precision": FP32,
         "warm": "previous", "tol": 1e-8, "pre": 1, "post": 2, "cpre": -1, "cpost": -1, "steps": 3},
        # the largest single-GPU configuration, with the cycle the benchmark sets
        {"name": "wide3d_512x256x256_fp32", "kind": "step", "flow": "wide3d", "n": "512x256x256", "precision": FP32,
         "warm": "previous", "tol": 1e-8, "pre": 1, "post": 1, "cpre": 2, "cpost": 2, "steps": 6},
        # a sweep over angle, slip length, capillary number and density ratio: 64 uneven 2D grids
        {"name": "sweep2d_64_fp32", "kind": "sweep", "count": 64, "precision": FP32, "tol": 1e-8, "steps": 2},
        # the network on a small ragged grid: a prediction bound by launches
        {"name": "unet_forward_40x24x16", "kind": "forward", "n": "40x24x16"},
        # a prediction at the size of an ordinary 3D run
        {"name": "unet_forward_128", "kind": "forward", "n": "128x128x128"},
        # and at the size the benchmark quotes inference on
        {"name": "unet_forward_256", "kind": "forward", "n": "256x256x256"},
        # one training step at the size the network is trained on
        {"name": "unet_train_64", "kind": "train", "n": "64x64x64"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, dim, least, most):
    """Extents that coarsen by 2 to at most 64 cells, with about a log-uniform cell count."""
    target = _log(rng, least, most)
    for _ in range(10000):
        k = rng.randint(3, 7 if dim == 2 else 6)
        f = [rng.randint(2, 12) for _ in range(dim)]
        if math.prod(f) > 64 or max(f) > 5 * min(f):
            continue
        n = [v << k for v in f]
        if 0.8 * target <= math.prod(n) <= 1.25 * target and math.prod(n) <= most and max(n) <= 512:
            return "x".join(str(v) for v in n)
    return "128x64" if dim == 2 else "64x64x64"


def draw(rng):
    kind = rng.choice(["step2d", "step2d", "step3d", "step3d", "sweep", "forward", "forward", "train"])
    if kind in ("step2d", "step3d"):
        dim = 2 if kind == "step2d" else 3
        precision = rng.choice([FP64, FP32])
        n = _grid(rng, dim, *((2048, 131072) if dim == 2 else (32768, 16777216 if precision == FP32 else 1048576)))
        return {"kind": "step", "flow": rng.choice(["drop2d", "couette2d"]) if dim == 2 else "drop3d", "n": n,
                "precision": precision, "warm": rng.choice(["previous", "extrapolated"]),
                "tol": 1e-12 if precision == FP64 else 1e-8, "pre": rng.randint(1, 2), "post": rng.randint(1, 2),
                "cpre": -1, "cpost": -1, "steps": rng.randint(1, 4)}
    if kind == "sweep":
        return {"kind": "sweep", "count": int(_log(rng, 8, 65)), "precision": FP32, "tol": 1e-8,
                "steps": rng.randint(1, 2)}
    if kind == "forward":
        return {"kind": "forward", "n": "x".join(str(8 * int(_log(rng, 1, 28.5))) for _ in range(3))}
    return {"kind": "train", "n": "x".join(str(8 * int(_log(rng, 1, 11.5))) for _ in range(3))}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _extents(case):
    return tuple(int(v) for v in case["n"].split("x"))


def _cap(n, h, L, R, theta, centre, eps):
    """Tanh cap of contact angle theta on the low wall of the last axis (the fields of inputs.py, on the GPU)."""
    axes = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) * h for m in n]
    r2 = (axes[-1] + R * math.cos(theta)).square()
    for a in reversed(range(len(n) - 1)):
        r2 = r2[..., None] + (axes[a] - centre[a] * L[a]).square()
    return 0.5 * (1.0 + torch.tanh((R - r2.sqrt()) / (2.0 * eps)))


def _workload(flow, n, seed):
    """Parameter set and initial phase field of one run: the flows of inputs.py with seeded angle, place and size."""
    r = random.Random(seed)
    if flow == "couette2d":
        nx, ny = n
        h = 1.0 / ny
        L, U, mu = (nx * h, 1.0), 0.1, 0.1
        x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * h
        x1, x2 = (0.25 + r.uniform(-0.05, 0.05)) * L[0], (0.75 + r.uniform(-0.05, 0.05)) * L[0]
        row = 0.5 * (torch.tanh((x - x1) / (2 * h)) + torch.tanh((x2 - x) / (2 * h)))
        p = dict(rho1=1.0, rho2=1.0, mu1=mu, mu2=mu, sigma=mu * U / 0.05, eps=h, gamma=2.5 * U,
                 theta_eq=math.radians(r.uniform(80, 100)), slip_length=h, U_lo=-U, U_hi=U)
        phi = row.expand(ny, nx).contiguous()
    elif flow == "drop2d":
        nx, ny = n
        h = 1.0 / nx
        L = (1.0, ny * h)
        R = min(0.4 * L[1], 0.2 * L[0]) * r.uniform(0.95, 1.05)
        p = dict(rho1=1.0, rho2=1.0, mu1=0.1, mu2=0.1, sigma=1.0, eps=h, gamma=1.0,
                 theta_eq=math.radians(r.uniform(50, 70)), slip_length=h, U_lo=0.0, U_hi=0.0)
        phi = _cap(n, h, L, R, math.pi / 2, (0.5 + r.uniform(-0.1, 0.1),), h)
    else:
        h = 1.0 / min(n)
        L = tuple(m * h for m in n)
        rho2, theta = (0.05, 45.0) if flow == "wide3d" else (0.1, 60.0)
        p = dict(rho1=1.0, rho2=rho2, mu1=0.05, mu2=0.005, sigma=1.0, eps=h, gamma=1.0,
                 theta_eq=math.radians(theta + r.uniform(-5, 5)), slip_length=h, U_lo=0.0, U_hi=0.0)
        # no cell noise: in FP32 it makes the first steps from rest too sensitive to rounding to be compared
        phi = _cap(n, h, L, 0.25 * r.uniform(0.95, 1.05), math.pi / 2,
                   (0.5 + r.uniform(-0.05, 0.05), 0.5 + r.uniform(-0.05, 0.05)), h)
    wl = inputs.Workload(flow, len(n), n, L, dt=0.0, steps=0, phi0=phi, **p)
    wl.dt = inputs.stable_dt(wl)
    return wl


def _sweep(case, seed):
    """The first instances of inputs.sweep_2d with seeded angle, slip length, density ratio and surface tension."""
    r, out = random.Random(seed), []
    for w in inputs.sweep_2d(n_inst=case["count"]):
        w = dataclasses.replace(w, theta_eq=math.radians(r.uniform(30, 150)), slip_length=r.uniform(0.5, 4) * w.h,
                                rho1=r.uniform(1, 20), sigma=w.sigma * r.uniform(0.8, 1.25),
                                phi0=torch.from_numpy(w.phi0))
        w.dt = inputs.stable_dt(w)
        out.append(w)
    return out


def _pinned(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True)


def _solver(wl, case, phi):
    s = cdi.Solver(wl.dim, wl.n, wl.L, cdi.FP64 if case["precision"] == FP64 else cdi.FP32_MIXED)
    s.set_fluids(wl.rho1, wl.rho2, wl.mu1, wl.mu2, wl.sigma, wl.eps, wl.gamma)
    s.set_wall(cdi.WALL_LO, wl.theta_eq, wl.slip_length, wl.U_lo)
    s.set_wall(cdi.WALL_HI, wl.theta_eq, wl.slip_length, wl.U_hi)
    s.set_phi(phi.numpy())
    return s


def _net_fields(n, seed):
    """(f / rms(f), rho / max(rho)) of a drop whose forcing sits at the interface, and a smooth target."""
    wl = _workload("drop3d", n, seed)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    f = torch.randn(wl.phi0.shape, generator=g, dtype=torch.float64, device="cuda")
    f = f * (0.05 + 4.0 * wl.phi0 * (1.0 - wl.phi0))
    f = (f - f.mean()) / (f - f.mean()).square().mean().sqrt()
    x = torch.stack([f, (wl.rho1 - wl.rho2) * wl.phi0 + wl.rho2], dim=-1)
    c = [torch.arange(m, dtype=torch.float64, device="cuda") / m for m in n]
    k = torch.randn(3, generator=g, dtype=torch.float64, device="cuda").tolist()
    t = (torch.cos(math.pi * c[2])[:, None, None] * k[0] + torch.sin(2 * math.pi * c[1])[:, None] * k[1]
         + torch.sin(2 * math.pi * c[0]) * k[2]) + 0.5 * wl.phi0
    return x, t


def prepare(case, seed):
    if case["kind"] == "step":
        wl = _workload(case["flow"], _extents(case), seed)
        phi = _pinned(wl.phi0.shape).copy_(wl.phi0)
        s = _solver(wl, case, phi)
        s.set_smoothing(case["pre"], case["post"])
        s.set_coarse_smoothing(case["cpre"], case["cpost"])
        s.set_solver(case["tol"], 100, cdi.WARM_EXTRAP if case["warm"] == "extrapolated" else cdi.WARM_PREV)
        out = [_pinned(s.cell_shape)] + [_pinned(s.face_shape(a)) for a in range(s.dim)] + [_pinned(s.cell_shape)]
        return {"case": case, "solver": s, "dt": wl.dt, "out": out, "views": [o.numpy() for o in out],
                "snap": [torch.empty(o.shape) for o in out] if case["precision"] == FP32 else None}
    if case["kind"] == "sweep":
        wls = _sweep(case, seed)
        solvers = []
        for w in wls:
            s = _solver(w, case, w.phi0)
            s.set_smoothing(2, 2)
            s.set_solver(case["tol"], 100, cdi.WARM_EXTRAP)
            solvers.append(s)
        batch = cdi.Batch(solvers)
        batch.set_threads(1024)
        # every instance's phi, u, v, p in one flat buffer a field
        sizes = [[math.prod(s.cell_shape), math.prod(s.face_shape(0)), math.prod(s.face_shape(1)),
                  math.prod(s.cell_shape)] for s in solvers]
        out = [_pinned(sum(z[k] for z in sizes)) for k in range(4)]
        views, at = [], [0, 0, 0, 0]
        for s, z in zip(solvers, sizes):
            shapes = [s.cell_shape, s.face_shape(0), s.face_shape(1), s.cell_shape]
            v = [out[k][at[k]:at[k] + z[k]].view(shapes[k]).numpy() for k in range(4)]
            at = [a + b for a, b in zip(at, z)]
            views.append((v[0], [v[1], v[2]], v[3]))
        return {"case": case, "solvers": solvers, "batch": batch, "dt": np.array([w.dt for w in wls]), "out": out,
                "views": views, "snap": [torch.empty(o.shape) for o in out]}
    n = _extents(case)
    net = cdi.Unet(n)
    net.set_params(inputs.unet_initial_params(seed))
    x, t = _net_fields(n, seed)
    if case["kind"] == "forward":
        x = x.to(torch.float32).contiguous()
        return {"case": case, "net": net, "x": x, "y": torch.empty(x.shape[:3], device="cuda")}
    return {"case": case, "net": net, "x": x.cpu().numpy(), "t": t.cpu().numpy()}


def run(state):
    kind = state["case"]["kind"]
    if kind == "step":
        s, v = state["solver"], state["views"]
        s.step(state["dt"], state["case"]["steps"])
        s.get_fields(out=(v[0], v[1:-1], v[-1]))
        answer = list(state["out"])
        if state["snap"] is not None:
            answer = [a.copy_(b) for a, b in zip(state["snap"], answer)]
        if state["case"]["flow"] == "drop2d":
            answer += list(s.contact_angle(cdi.WALL_LO))
        return answer
    if kind == "sweep":
        state["batch"].step(state["dt"], state["case"]["steps"])
        for s, v in zip(state["solvers"], state["views"]):
            s.get_fields(out=v)
        return [a.copy_(b) for a, b in zip(state["snap"], state["out"])]
    if kind == "forward":
        state["net"].forward_device(state["x"], state["y"])
        return state["y"]
    loss, grads = state["net"].train_step(state["x"], state["t"], lr=1e-3, want_grads=True)
    return {"loss": loss, "grads": grads.astype(np.float32)}


def work(case):
    """Steps: each RK stage reads phi and the velocity and writes both, and its pressure solve reads and writes p
    (8 bytes a cell in both forms); the read-out writes every field once.  Network: the convolutions' operations, its
    input, output and parameters."""
    if case["kind"] in ("step", "sweep"):
        if case["kind"] == "step":
            grids = [_extents(case)]
        else:
            grids = [w.n for w in _sweep(case, 1)]
        word = 8 if case["precision"] == FP64 else 4
        cells, dim = sum(math.prod(n) for n in grids), len(grids[0])
        state = (1 + dim) * word
        stage = 2 * state + 2 * 8
        return {"bytes": cells * (4 * case["steps"] * stage + (2 + dim) * 8), "flops": 0}
    n = _extents(case)
    cells = math.prod(n)
    flops = 0
    for (_, ci, co, taps), level in zip(inputs.UNET_LAYERS, (0, 1, 2, 3, 2, 1, 0, 0)):
        flops += 2 * taps * ci * co * (cells >> (3 * level))
    params = sum(t * ci * co + co for _, ci, co, t in inputs.UNET_LAYERS)
    if case["kind"] == "forward":
        return {"bytes": 12 * cells + 2 * params, "flops": flops}
    return {"bytes": 24 * cells + 4 * 8 * params, "flops": 3 * flops}


# --------------------------------------------------------------------------
# the same results in plain FP64 torch
# --------------------------------------------------------------------------

class _Plain:
    """The time step of the paper in FP64 torch: a 2D grid is a 3D one of a single row in y, walls at both ends of z.
    Velocity components sit on the low faces of their cells; w has nz + 1 planes."""

    DELTA = TAU = 1e-6

    def __init__(self, wl):
        self.wl, self.dim = wl, wl.dim
        n = wl.n if wl.dim == 3 else (wl.n[0], 1, wl.n[1])
        self.shape, self.h = (n[2], n[1], n[0]), wl.L[0] / wl.n[0]
        self.phi = wl.phi0.to("cuda", torch.float64).reshape(self.shape)
        self.u = [torch.zeros(self.shape, dtype=torch.float64, device="cuda") for _ in range(2)]
        self.u.append(torch.zeros((n[2] + 1, n[1], n[0]), dtype=torch.float64, device="cuda"))
        self.p = torch.zeros_like(self.phi)
        # eigenvalues of the five/seven point Laplacian; z extended evenly to twice its length
        lam = []
        for m, half in ((2 * n[2], False), (n[1], False), (n[0], True)):
            k = torch.arange(m // 2 + 1 if half else m, dtype=torch.float64, device="cuda")
            lam.append((2.0 * torch.cos(2.0 * math.pi * k / m) - 2.0) / self.h ** 2)
        self.lam = lam[0][:, None, None] + lam[1][:, None] + lam[2]
        self.lam[0, 0, 0] = 1.0

    @staticmethod
    def lo(q, axis):  # value of the low neighbour along a periodic axis (0: x, 1: y)
        return torch.roll(q, 1, 2 - axis)

    @staticmethod
    def hi(q, axis):
        return torch.roll(q, -1, 2 - axis)

    def d12(self, s, axis):
        h = self.h
        if axis < 2:
            a, b = self.lo(s, axis), self.hi(s, axis)
            return (b - a) / (2 * h), (b - 2 * s + a) / h ** 2
        d1, d2 = torch.empty_like(s), torch.empty_like(s)
        d1[1:-1] = (s[2:] - s[:-2]) / (2 * h)
        d2[1:-1] = (s[2:] - 2 * s[1:-1] + s[:-2]) / h ** 2
        d1[0] = (-3 * s[0] + 4 * s[1] - s[2]) / (2 * h)
        d1[-1] = (3 * s[-1] - 4 * s[-2] + s[-3]) / (2 * h)
        d2[0] = (2 * s[0] - 5 * s[1] + 4 * s[2] - s[3]) / h ** 2
        d2[-1] = (2 * s[-1] - 5 * s[-2] + 4 * s[-3] - s[-4]) / h ** 2
        return d1, d2

    def psi(self, phi):
        pt = phi.clamp(self.DELTA, 1 - self.DELTA)
        return pt, self.wl.eps * torch.log(pt / (1 - pt))

    def wall(self, phi, psi, u, side):
        """Ghost values of u and v and the wall viscosities on one wall (Model 4A)."""
        wl, h = self.wl, self.h
        rows = slice(0, 4) if side == 0 else slice(-4, None)
        ph, ps = phi[rows], psi[rows]
        if side == 1:
            ph, ps = ph.flip(0), ps.flip(0)  # the rows from the wall inwards: normal derivatives along the inward normal
        g, lap = [], 0.0
        for a in range(3):
            d1, d2 = self.d12(ps, a)
            g.append(d1[:2])
            lap = lap + d2[:2]
        g2 = g[0] ** 2 + g[1] ** 2 + g[2] ** 2
        pt = ph[:2].clamp(self.DELTA, 1 - self.DELTA)
        kap = (1 - 2 * pt) * (1 - g2) / wl.eps - lap
        if self.dim == 3:  # less the normal curvature along the contact line
            s = ps[:2]
            px, py = g[0], g[1]
            pxx, pyy = self.d12(ps, 0)[1][:2], self.d12(ps, 1)[1][:2]
            ax, bx = self.hi(s, 0), self.lo(s, 0)
            pxy = (self.hi(ax, 1) - self.lo(ax, 1) - self.hi(bx, 1) + self.lo(bx, 1)) / (4 * h ** 2)
            num = py * py * pxx - 2 * px * py * pxy + px * px * pyy
            kap = kap + num / ((px * px + py * py + self.TAU ** 2) * (g2.sqrt() + self.TAU))
        ext = lambda q: 0.5 * (3 * q[0] - q[1])  # noqa: E731
        phw, psw, dnw, kw = ext(ph).clamp(0, 1), ext(ps), ext(g[2]), ext(kap)
        ghost, visc = [], []
        for a in range(2):
            low = lambda q: torch.roll(q, 1, 1 - a)  # noqa: E731
            mean = lambda q: 0.5 * (q + low(q))  # noqa: E731
            pb = mean(phw)
            P = pb * (1 - pb)
            muw = (wl.mu1 - wl.mu2) * pb + wl.mu2
            beta = muw / wl.slip_length
            dtau = (psw - low(psw)) / h
            slip = -(6 * wl.sigma / beta) * (P * mean(dnw) + P * (1 + mean(kw) * mean(psw)) * math.cos(wl.theta_eq)) * (
                P / wl.eps * dtau)
            lw = wl.slip_length / h
            U = (wl.U_lo if side == 0 else wl.U_hi) if a == 0 else 0.0
            uf = u[a][0 if side == 0 else -1]
            ghost.append((U + slip - uf * (0.5 - lw)) / (0.5 + lw))
            visc.append(muw)
        return ghost, visc

    def rhs(self, phi, u):
        wl, h = self.wl, self.h
        pt, psi = self.psi(phi)
        g, lap = [], 0.0
        for a in range(3):
            d1, d2 = self.d12(psi, a)
            g.append(d1)
            lap = lap + d2
        g2 = g[0] ** 2 + g[1] ** 2 + g[2] ** 2
        P = pt * (1 - pt)
        muc = 6 * wl.sigma * (P * (1 - 2 * pt) * (1 - g2) / wl.eps - P * lap)
        nrm = [q / (g2.sqrt() + self.TAU) for q in g]
        walls = [self.wall(phi, psi, u, s) for s in (0, 1)]

        def flux(L, R, nL, nR, uf):
            pb = 0.5 * (L + R)
            pc = pb.clamp(self.DELTA, 1 - self.DELTA)
            return uf * pb - wl.gamma * (wl.eps * (R - L) / h - pc * (1 - pc) * 0.5 * (nL + nR))

        drho, m, rphi = wl.rho1 - wl.rho2, [], 0.0
        for a in range(2):
            F = flux(self.lo(phi, a), phi, self.lo(nrm[a], a), nrm[a], u[a])
            m.append(drho * F + wl.rho2 * u[a])
            rphi = rphi - (self.hi(F, a) - F) / h
        F = torch.zeros_like(u[2])
        F[1:-1] = flux(phi[:-1], phi[1:], nrm[2][:-1], nrm[2][1:], u[2][1:-1])
        mz = drho * F + wl.rho2 * u[2]
        mz[0] = mz[-1] = 0.0
        m.append(mz)
        rphi = rphi - (F[1:] - F[:-1]) / h
        mu = (wl.mu1 - wl.mu2) * phi + wl.mu2

        def edge(a, b):
            """Momentum flux and stress of the edges between a- and b-faces, both tangential axes."""
            conv = 0.25 * (m[b] + self.lo(m[b], a)) * (u[a] + self.lo(u[a], b))
            me = 0.25 * (mu + self.lo(mu, a) + self.lo(mu, b) + self.lo(self.lo(mu, a), b))
            return me * ((u[a] - self.lo(u[a], b)) / h + (u[b] - self.lo(u[b], a)) / h) - conv

        def edge_z(a):
            """Edges between a-faces and the interior z-faces."""
            wm = 0.5 * (m[2] + self.lo(m[2], a))[1:-1]
            ua = 0.5 * (u[a][:-1] + u[a][1:])
            mm = mu + self.lo(mu, a)
            me = 0.25 * (mm[:-1] + mm[1:])
            tau = me * ((u[a][1:] - u[a][:-1]) / h + (u[2] - self.lo(u[2], a))[1:-1] / h)
            return tau, wm * ua, ua

        r = []
        for a in range(2):
            C = 2 * mu * (self.hi(u[a], a) - u[a]) / h - 0.25 * (m[a] + self.hi(m[a], a)) * (u[a] + self.hi(u[a], a))
            v = (C - self.lo(C, a)) / h
            E = edge(a, 1 - a)
            v = v + (self.hi(E, 1 - a) - E) / h
            tau, conv, _ = edge_z(a)
            full = torch.zeros_like(u[2])
            full[1:-1] = tau - conv
            full[0] = walls[0][1][a] * (u[a][0] - walls[0][0][a]) / h
            full[-1] = walls[1][1][a] * (walls[1][0][a] - u[a][-1]) / h
            v = v + (full[1:] - full[:-1]) / h
            r.append(v + 0.5 * (muc + self.lo(muc, a)) * (phi - self.lo(phi, a)) / h)
        C = 2 * mu * (u[2][1:] - u[2][:-1]) / h - 0.25 * (m[2][1:] + m[2][:-1]) * (u[2][1:] + u[2][:-1])
        v = (C[1:] - C[:-1]) / h
        for b in range(2):
            tau = edge_z(b)[0]
            conv = 0.25 * (m[b][:-1] + m[b][1:]) * (u[2] + self.lo(u[2], b))[1:-1]
            E = tau - conv
            v = v + (self.hi(E, b) - E) / h
        rz = torch.zeros_like(u[2])
        rz[1:-1] = v + 0.5 * (muc[:-1] + muc[1:]) * (phi[1:] - phi[:-1]) / h
        r.append(rz)
        return rphi, r

    def rho_faces(self, phi):
        rho = (self.wl.rho1 - self.wl.rho2) * phi + self.wl.rho2
        f = [0.5 * (rho + self.lo(rho, a)) for a in range(2)]
        z = torch.ones_like(self.u[2])
        z[1:-1] = 0.5 * (rho[1:] + rho[:-1])
        return f + [z]

    def grad(self, p):
        g = [(p - self.lo(p, a)) / self.h for a in range(2)]
        z = torch.zeros_like(self.u[2])
        z[1:-1] = (p[1:] - p[:-1]) / self.h
        return g + [z]

    def div(self, u):
        d = (u[2][1:] - u[2][:-1]) / self.h
        for a in range(2):
            d = d + (self.hi(u[a], a) - u[a]) / self.h
        return d

    def poisson(self, f):
        """Constant-coefficient solve by FFT, the wall axis extended evenly."""
        k = torch.fft.rfftn(torch.cat([f, f.flip(0)], 0)) / self.lam
        k[0, 0, 0] = 0.0
        return torch.fft.irfftn(k, s=(2 * f.shape[0],) + tuple(f.shape[1:]))[:f.shape[0]]

    def solve(self, beta, f, p):
        """Preconditioned conjugate gradients for div(beta grad p) = f."""
        A = lambda q: self.div([b * d for b, d in zip(beta, self.grad(q))])  # noqa: E731
        f = f - f.mean()
        p = p - p.mean()
        r = f - A(p)
        stop = 1e-14 * float(f.norm())
        z = self.poisson(r)
        d, rz = z, (r * z).sum()
        for _ in range(150):
            if float(r.norm()) <= stop:
                break
            q = A(d)
            alpha = rz / (d * q).sum()
            p = p + alpha * d
            r = r - alpha * q
            z = self.poisson(r)
            new = (r * z).sum()
            d = z + (new / rz) * d
            rz = new
        return p - p.mean()

    def step(self, dt):
        phi0, u0 = self.phi, self.u
        phi, u = phi0, u0
        rf0 = self.rho_faces(phi0)
        for k, (b, c) in enumerate(((1 / 6, 0.5), (1 / 3, 0.5), (1 / 3, 1.0), (1 / 6, 1.0))):
            rphi, rm = self.rhs(phi, u)
            if k == 0:
                aphi, am = b * rphi, [b * q for q in rm]
            else:
                aphi, am = aphi + b * rphi, [s + b * q for s, q in zip(am, rm)]
            phi = phi0 + dt * (aphi if k == 3 else c * rphi)
            rf = self.rho_faces(phi)
            u = [(r0 * v + dt * (s if k == 3 else c * q)) / r1 for r0, v, s, q, r1 in zip(rf0, u0, am, rm, rf)]
            beta = [1.0 / q for q in rf]
            self.p = self.solve(beta, self.div(u) / (c * dt), self.p)
            u = [v - c * dt * q * g for v, q, g in zip(u, beta, self.grad(self.p))]
            u[2][0] = u[2][-1] = 0.0
        self.phi, self.u = phi, u

    def fields(self):
        if self.dim == 3:
            return [self.phi, self.u[0], self.u[1], self.u[2], self.p]
        return [q[:, 0].contiguous() for q in (self.phi, self.u[0], self.u[2], self.p)]

    def contact_angle(self):
        """2D, low wall: mean angle of the two crossings of phi_w = 1/2, and their distance."""
        _, psi = self.psi(self.phi)
        g = self.d12(psi, 2)[0]
        ext = lambda q: (0.5 * (3 * q[0] - q[1]))[0].cpu().numpy()  # noqa: E731
        phw, psw, gn = np.clip(ext(self.phi), 0, 1), ext(psi), ext(g)
        gt = (np.roll(psw, -1) - np.roll(psw, 1)) / (2 * self.h)
        nx, i0, x, th = len(phw), int(np.argmin(phw)), [], []
        for k in range(nx):
            i, j = (i0 + k) % nx, (i0 + k + 1) % nx
            if (phw[i] < 0.5) != (phw[j] < 0.5):
                t = (0.5 - phw[i]) / (phw[j] - phw[i])
                n, s = gn[i] + t * (gn[j] - gn[i]), gt[i] + t * (gt[j] - gt[i])
                x.append((i0 + k + 0.5 + t) * self.h)
                th.append(math.acos(max(-1.0, min(1.0, -n / math.hypot(n, s)))))
        return [0.5 * (th[0] + th[1]), x[1] - x[0]]


def _net_exact(case, seed):
    """The network in FP64: convolutions as sums of shifted products, gradients by autograd."""
    n = _extents(case)
    flat = torch.from_numpy(inputs.unet_initial_params(seed)).to("cuda").float().double()
    flat.requires_grad_(case["kind"] == "train")
    par, at = {}, 0
    for name, ci, co, taps in inputs.UNET_LAYERS:
        w = flat[at:at + taps * co * ci].view(taps, co, ci)
        at += taps * co * ci
        par[name] = (w, flat[at:at + co])
        at += co
    x, t = _net_fields(n, seed)
    x = x.float().double().permute(3, 0, 1, 2)

    def conv(q, name, relu=True):
        w, b = par[name]
        nz, ny, nx = q.shape[1:]
        y = b[:, None]
        if w.shape[0] == 1:
            return (y + w[0] @ q.reshape(q.shape[0], -1)).view(-1, nz, ny, nx)
        pad = torch.nn.functional.pad(q, (1, 1, 1, 1, 1, 1))
        for k in range(27):
            z, r, c = k // 9, (k // 3) % 3, k % 3
            y = y + w[k] @ pad[:, z:z + nz, r:r + ny, c:c + nx].reshape(q.shape[0], -1)
        return (y.relu() if relu else y).view(-1, nz, ny, nx)

    pool = lambda q: torch.nn.functional.avg_pool3d(q[None], 2)[0]  # noqa: E731
    up = lambda q: q.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    e0 = conv(x, "e0")
    e1 = conv(pool(e0), "e1")
    e2 = conv(pool(e1), "e2")
    d2 = conv(torch.cat([up(conv(pool(e2), "b")), e2]), "d2")
    d1 = conv(torch.cat([up(d2), e1]), "d1")
    y = conv(conv(torch.cat([up(d1), e0]), "d0"), "head")[0]
    if case["kind"] == "forward":
        return y
    loss = (y - t).square().mean()
    return {"loss": float(loss.detach()), "grads": torch.autograd.grad(loss, flat)[0]}


def exact(case, seed):
    if case["kind"] in ("forward", "train"):
        return _net_exact(case, seed)
    if case["kind"] == "sweep":
        wls = _sweep(case, seed)
        if sum(math.prod(w.n) for w in wls) * case["steps"] > 2.5e7:
            return None
        parts = []
        for w in wls:
            m = _Plain(w)
            for _ in range(case["steps"]):
                m.step(w.dt)
            parts.append([f.reshape(-1) for f in m.fields()])
        return [torch.cat(f) for f in zip(*parts)]
    wl = _workload(case["flow"], _extents(case), seed)
    if math.prod(wl.n) * case["steps"] > 6e7:  # the largest grid: over 20 seconds
        return None
    m = _Plain(wl)
    for _ in range(case["steps"]):
        m.step(wl.dt)
    return m.fields() + (m.contact_angle() if case["flow"] == "drop2d" else [])
