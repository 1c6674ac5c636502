"""Performance cases of the DD-CCLB steppers and of the discrete adjoint.

Each case is one call sequence of a user's program: make a simulation from
host fields, then, per pass, advance it and take the result (the state saved
to a device buffer, a snapshot of the fields, or the gradients).  ``exact``
gives the same results in plain 64-bit torch, written from the equations of
arXiv 2311.10314 and the stepper's documented conventions.

Kinds of case:
  step2d     ``Sim.step`` then ``Sim.save_state`` into a buffer the program
             keeps (restart files, slab exchange, adjoint checkpoints)
  monitor2d  ``Sim.step`` then ``Sim.fields`` and ``Sim.mass`` (what a
             program prints, plots or tests for equilibrium)
  step3d     ``Sim3D.step`` then reads of C_i, u and P into a snapshot kept
             in the step's precision
  adjoint    ``adjoint.rollout`` and ``backward``: the x-centroid of a drop
             after T steps and its gradients (create, forward, reverse sweep)
"""
import math

import numpy as np
import torch

import paper_2311_10314_gb300 as ddcc
from paper_2311_10314_gb300 import _lib, adjoint

SOLID_XI = 3.0 / math.sqrt(2.0)     # solid layer eps0 = 6
PSI_MIN = 1e-6


def listed():
    return [
        # the smallest grid in use: a drop on a flat wall, double precision,
        # a few steps between saves (launch latency and one wave of blocks)
        dict(name="wall_64_f64", kind="step2d", scene="wall", nx=64, ny=64, phases=2, f64=True, field=False, steps=10),
        # three-phase lens among solid circles at 256^2, single precision
        dict(name="porous_256_f32", kind="step2d", scene="porous", nx=256, ny=256, phases=3, f64=False, field=False,
             steps=50),
        # the ternary compound drop of the spreading tables, double precision,
        # with a full read-out of fields and masses (odd aspect, walls in y)
        dict(name="compound_300x170_f64", kind="monitor2d", scene="wall", nx=300, ny=170, phases=3, f64=True,
             field=False, steps=10),
        # a channel between two wavy walls with inflow and outflow
        dict(name="channel_150_f32", kind="step2d", scene="channel", nx=150, ny=150, phases=3, f64=False, field=False,
             steps=40),
        # an emulsion driven through a porous matrix at 1024^2, ragged in x
        dict(name="emulsion_1021x1024_f32", kind="step2d", scene="porous", nx=1021, ny=1024, phases=3, f64=False,
             field=False, steps=20),
        # four phases in a porous medium, angles per circle, double precision
        dict(name="imbibition_512_f64", kind="step2d", scene="porous", nx=512, ny=512, phases=4, f64=True, field=True,
             steps=4),
        # the production run: four phases imbibing a porous medium, 4096^2
        dict(name="imbibition_4096_f32", kind="step2d", scene="porous", nx=4096, ny=4096, phases=4, f64=False,
             field=True, steps=10),
        # compound drop on a solid sphere, single precision, the largest box
        # (the snapshot goes through host memory, so it is taken seldom)
        dict(name="sphere_208x192x160_f32", kind="step3d", nx=208, ny=192, nz=160, phases=3, f64=False, field=False,
             steps=200),
        # a ragged 3D box with one drop and per-node angles
        dict(name="sphere_101x77x63_f32", kind="step3d", nx=101, ny=77, nz=63, phases=2, f64=False, field=True,
             steps=40),
        # the 3D step in double precision
        dict(name="sphere_96x80x72_f64", kind="step3d", nx=96, ny=80, nz=72, phases=3, f64=True, field=False, steps=10),
        # gradients of a drop's centroid on a wavy wall, single precision,
        # with a checkpoint every 25 steps
        dict(name="adjoint_256_f32", kind="adjoint", scene="wall", nx=256, ny=256, phases=2, f64=False, field=True,
             steps=100, ckpt=25),
        # the double-precision gradient on a small ragged grid, three phases
        dict(name="adjoint_130x94_f64", kind="adjoint", scene="wall", nx=130, ny=94, phases=3, f64=True, field=True,
             steps=24, ckpt=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step2d", "step2d", "step2d", "step2d", "monitor2d", "step3d", "step3d", "adjoint"])
    f64 = rng.random() < 0.4
    phases = rng.choice([2, 3, 4])
    if kind == "step3d":
        nx, ny, nz = (_log_int(rng, 20, 128 if f64 else 224) for _ in range(3))
        if rng.random() < 0.5:
            nx = max(20, nx // 4 * 4)
        cap = 64 ** 3 if f64 else 192 ** 3
        while nx * ny * nz > cap:
            ny, nz = max(16, ny * 3 // 4), max(16, nz * 3 // 4)
            nx = nx if nx * 256 <= cap else nx // 2
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, phases=phases, f64=f64, field=rng.random() < 0.5,
                    steps=rng.randint(4, 8) if f64 else rng.randint(10, 40))
    if kind == "adjoint":
        nx, ny = _log_int(rng, 64, 200 if f64 else 600), _log_int(rng, 64, 160 if f64 else 400)
        steps = rng.randint(8, 20) if f64 else rng.randint(20, 80)
        return dict(kind=kind, scene="wall", nx=nx, ny=ny, phases=rng.choice([2, 2, 3]), f64=f64, field=True,
                    steps=steps, ckpt=rng.randint(4, 20))
    scene = rng.choice(["wall", "porous", "porous", "channel"])
    if kind == "monitor2d":
        f64 = True
    top = 512 if scene != "porous" else (700 if f64 else 3000)
    nx, ny = _log_int(rng, 48, top), _log_int(rng, 64, top)
    return dict(kind=kind, scene=scene, nx=nx, ny=ny, phases=phases, f64=f64, field=scene != "channel" and
                rng.random() < 0.5, steps=rng.randint(4, 10) if f64 else rng.randint(8, 40))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _params(case, nx, ny, N):
    """Physical parameters in lattice units; the multiphase settings keep the
    derived phase bounded at triple regions (small mobility and eta)."""
    tau, d0 = 0.8, 1.0 / 3.0
    prm = dict(nx=nx, ny=ny, nphase=N, periodic_x=1, periodic_y=1, rho=[1.0] * N, nu=[(tau - 0.5) * d0] * N,
               width=4.0 if N == 2 else 8.0, eps0=2.0 * math.sqrt(2.0) * SOLID_XI, d0=d0, m0=(tau - 0.5) * d0,
               eta=[1.0] * (N - 1), s_f=[1.0, 1.2, 1.2, 1.2, 1.2], s_g=[1.0, 1.2, 1.2, 1.2], rho0=1.0,
               body_force=(0.0, 0.0))
    sigma = 0.01 if N == 2 else 0.005
    prm["sigma"] = [[0.0 if i == j else sigma for j in range(N)] for i in range(N)]
    if N > 2:
        prm["m0"] = 0.01
        prm["eta"] = [0.1] * (N - 1)
    if case.get("scene") == "porous":
        prm["rho"] = [1.0, 0.8, 0.5, 0.1][:N]
        prm["body_force"] = (1e-6, 0.0)
    elif case.get("scene") == "channel":
        prm["periodic_x"] = prm["periodic_y"] = 0
        prm["d0"] = d0 = 0.3
        prm["nu"] = [(tau - 0.5) * d0] * N
        if N > 2:
            prm["rho"] = [1.0] * (N - 1) + [0.1]
            prm["eta"] = [0.01 / ((tau - 0.5) * d0)] * (N - 1)
    elif case["kind"] == "step3d":
        prm["nz"] = case["nz"]
        prm["d0"] = 0.4
        prm["s_f"], prm["s_g"] = [1.0, 1.0], [1.0, 1.2, 1.2, 0.8]
        prm["nu"] = [(tau - 0.5) * 0.4] * N
        prm["body_force"] = (0.0, 0.0, 0.0)
        prm["sigma"] = [[0.0 if i == j else 0.01 for j in range(N)] for i in range(N)]
        if N == 2:
            prm["m0"] = (tau - 0.5) * 0.4
    else:
        prm["periodic_y"] = 0
        if N > 2:
            prm["nu"] = [0.1] * N
    return prm


def _profile(dist, width):
    """1 inside (dist < 0), 0 outside, over an interface of this width."""
    return 0.5 * (1.0 - torch.tanh(2.0 * dist / width))


def _solid(d):
    """Characteristic function of the distance from the solid (> 0 in the fluid)."""
    return torch.clamp(0.5 * (1.0 + torch.tanh(d / (math.sqrt(2.0) * SOLID_XI))), min=PSI_MIN)


def _circles(x, y, nx, ny, cell, lo, hi, rng):
    """Signed distance to the nearest of one circle per cell of a periodic
    jittered lattice, and that circle's number; radii in [lo, hi] x cell."""
    mx, my = max(1, round(nx / cell)), max(1, round(ny / cell))
    wx, wy = nx / mx, ny / my
    w = min(wx, wy)
    r = torch.as_tensor(rng.uniform(lo, hi, (my, mx)) * w, device=x.device)
    slack = 0.5 - hi
    cx = torch.as_tensor(rng.uniform(0.5 - slack, 0.5 + slack, (my, mx)), device=x.device)
    cy = torch.as_tensor(rng.uniform(0.5 - slack, 0.5 + slack, (my, mx)), device=x.device)
    ix, iy = torch.floor(x / wx).long(), torch.floor(y / wy).long()
    best = own = None
    for dj in (-1, 0, 1):
        for di in (-1, 0, 1):
            i, j = ix + di, iy + dj
            im, jm = i % mx, j % my
            d = torch.hypot(x - (i + cx[jm, im]) * wx, y - (j + cy[jm, im]) * wy) - r[jm, im]
            o = jm * mx + im
            if best is None:
                best, own = d, o
            else:
                own = torch.where(d < best, o, own)
                best = torch.minimum(best, d)
    return best, own, mx * my


def _inputs2d(case, seed):
    """Host fields of a two-dimensional scene: params, psi, C0 and the angles
    (uniform, per node, or per solid with the inflow of open ends)."""
    rng = np.random.default_rng([seed, case["nx"], case["ny"], case["phases"]])
    nx, ny, N = case["nx"], case["ny"], case["phases"]
    dev = _device()
    prm = _params(case, nx, ny, N)
    y, x = torch.meshgrid(torch.arange(ny, dtype=torch.float64, device=dev),
                          torch.arange(nx, dtype=torch.float64, device=dev), indexing="ij")
    out = dict(params=prm, cos=None, cos_field=None, walls=None, open_x=None)
    W = prm["width"]
    cos = np.cos(np.radians(rng.uniform(50.0, 130.0, N - 1)))
    if case["scene"] == "porous":
        d, own, n = _circles(x, y, nx, ny, max(48.0, min(96.0, min(nx, ny) / 6)), 0.25, 0.4, rng)
        psi = _solid(d)
        drop, which, m = _circles(x, y, nx, ny, max(40.0, min(120.0, min(nx, ny) / 4)), 0.2, 0.35, rng)
        phase = torch.as_tensor(rng.integers(0, N, m), device=dev)[which]
        c = _profile(drop, W)
        C0 = torch.stack([torch.where(phase == i, c, 0.0) for i in range(N - 1)])
        if case["field"]:
            ang = torch.as_tensor(np.cos(np.radians(rng.uniform(30.0, 150.0, (N - 1, n)))), device=dev)
            out["cos_field"] = ang[:, own].cpu().numpy()
        else:
            out["cos"] = cos
    elif case["scene"] == "channel":
        jit = rng.uniform(0.9, 1.1)
        U = 0.05 * ny * jit * torch.sqrt(x / nx) * torch.sin(3.0 * math.pi * x / nx)
        eps0 = prm["eps0"]
        psi1 = torch.clamp(0.5 + 0.5 * torch.tanh(2.0 * (y - ny / 4.0 + U) / eps0), min=PSI_MIN)
        psi2 = torch.clamp(0.5 - 0.5 * torch.tanh(2.0 * (y - 3.0 * ny / 4.0 - U) / eps0), min=PSI_MIN)
        psi = psi1 * psi2
        r = torch.hypot(x - nx * rng.uniform(0.45, 0.55), y - ny / 2.0)
        L = min(nx, ny)
        left, C = torch.ones_like(x), []
        for i in range(N - 1):
            c = _profile(r - L * (0.15 + 0.08 * i), W) * left
            C.append(c)
            left = left - c
        C0 = torch.stack(C)
        out["walls"] = [(psi1.cpu().numpy(), cos), (psi2.cpu().numpy(), cos[::-1].copy())]
        gap = np.clip((np.arange(ny) - ny / 4.0) * (3.0 * ny / 4.0 - np.arange(ny)), 0.0, None)
        out["open_x"] = (6.0 * 0.003 * gap / (ny / 2.0) ** 2, np.zeros((N - 1, ny)))
    else:
        wall = rng.uniform(0.15, 0.2) * ny
        amp = 0.03 * ny * (1.0 if case["field"] else 0.0)
        k = 2.0 * math.pi * max(1, round(nx / 64)) / nx
        yw = wall + amp * torch.sin(k * x)
        psi = _solid(y - yw)
        R = min(0.8 * (ny - wall) / 1.5, nx / (2.0 * N)) * rng.uniform(0.8, 0.95)
        xc = nx * rng.uniform(0.45, 0.55)
        C, left = [], torch.ones_like(x)
        for i in range(N - 1):
            r = torch.hypot(x - (xc + (i - (N - 2) / 2.0) * 1.6 * R), y - wall)
            c = _profile(r - R, W) * left
            C.append(c)
            left = left - c
        C0 = torch.stack(C)
        if case["field"]:
            c = torch.as_tensor(cos, device=dev)[:, None, None] + 0.1 * torch.sin(k * x + y / 7.0)
            out["cos_field"] = c.cpu().numpy()
        else:
            out["cos"] = cos
    out["psi"], out["C0"] = psi.cpu().numpy(), C0.cpu().numpy()
    return out


def _inputs3d(case, seed):
    """A compound drop on a solid sphere in a periodic box."""
    rng = np.random.default_rng([seed, case["nx"], case["ny"], case["nz"], case["phases"]])
    nx, ny, nz, N = case["nx"], case["ny"], case["nz"], case["phases"]
    dev = _device()
    prm = _params(case, nx, ny, N)
    L = min(nx, ny, nz)
    c = [n / 2.0 + rng.uniform(-0.5, 0.5) for n in (nx, ny, nz)]
    z, y, x = torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device=dev) for n in (nz, ny, nx)), indexing="ij")
    r = torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2)
    psi = _solid(r - 0.2 * L * rng.uniform(0.9, 1.1))
    W = prm["width"]
    drop = _profile(r - 0.33 * L, W) * _profile(c[1] - y, W)
    cuts = [1.0 - _profile(x - (c[0] + 0.15 * L * (i - (N - 3) / 2.0)), W) for i in range(N - 2)]
    C, left = [], drop
    for i in range(N - 1):
        part = left * (1.0 - cuts[i]) if i < N - 2 else left
        C.append(part)
        left = left - part
    cos = np.cos(np.radians(rng.uniform(60.0, 120.0, N - 1)))
    field = None
    if case["field"]:
        field = (torch.as_tensor(cos, device=dev)[:, None, None, None] + 0.1 * torch.sin(2.0 * math.pi * x / nx)
                 * torch.cos(2.0 * math.pi * z / nz)).cpu().numpy()
    return dict(params=prm, psi=psi.cpu().numpy(), C0=torch.stack(C).cpu().numpy(), cos=None if case["field"] else cos,
                cos_field=field)


# ----------------------------------------------------------------------------
# the calls
# ----------------------------------------------------------------------------

def prepare(case, seed):
    precision = ddcc.DDCC_FP64 if case["f64"] else ddcc.DDCC_FP32
    real = torch.float64 if case["f64"] else torch.float32
    st = dict(case=case, precision=precision, real=real)
    if case["kind"] == "step3d":
        inp = _inputs3d(case, seed)
        st["sim"] = ddcc.Sim3D(inp["params"], inp["psi"], inp["C0"], inp["cos"], inp["cos_field"], precision=precision)
        shape = (case["phases"] + 3,) + inp["psi"].shape
        st["host"] = torch.empty(shape, dtype=torch.float64, pin_memory=True)
        st["snapshot"] = st["host"] if case["f64"] else torch.zeros(shape, dtype=real)
        return st
    inp = _inputs2d(case, seed)
    if case["kind"] == "adjoint":
        st["inp"] = inp
        st["cos"] = torch.tensor(inp["cos_field"], dtype=real, device="cuda", requires_grad=True)
        st["psi"] = torch.tensor(inp["psi"], dtype=real, device="cuda", requires_grad=True)
        return st
    st["sim"] = sim = ddcc.Sim(inp["params"], inp["psi"], inp["C0"], inp["cos"], inp["cos_field"],
                               precision=precision, walls=inp["walls"], open_x=inp["open_x"])
    if case["kind"] == "step2d":
        N, nx, ny = case["phases"], case["nx"], case["ny"]
        st["buf"] = torch.zeros(sim.state_bytes(), dtype=torch.uint8, device="cuda")
        # the documented layout of a saved state: planes f (9 per phase), g, lagged
        org, pitch, plane = _lib.state_layout(nx, ny, N, 8 if case["f64"] else 4)
        planes = torch.as_strided(st["buf"].view(real), (11 * N + 3, ny, nx), (plane, pitch, 1), org)
        st["views"] = dict(f=planes[:9 * (N - 1)], g=planes[9 * (N - 1):9 * N], lag=planes[9 * N:])
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        inp, cos, psi = state["inp"], state["cos"], state["psi"]
        cos.grad = psi.grad = None
        J = adjoint.rollout(cos, psi, inp["params"], inp["C0"], case["steps"], ckpt=case["ckpt"],
                            precision=state["precision"])
        J.backward()
        return dict(J=J.detach().to(state["real"]), dJ_dcos=cos.grad, dJ_dpsi=psi.grad)
    sim = state["sim"]
    sim.step(case["steps"])
    if case["kind"] == "step2d":
        sim.save_state(state["buf"])
        return state["views"]
    if case["kind"] == "monitor2d":
        out = sim.fields()
        out["mass"] = sim.mass()
        return out
    ids = [ddcc.FIELD_C + i for i in range(case["phases"] - 1)]
    ids += [ddcc.FIELD_UX, ddcc.FIELD_UY, _lib.FIELD_UZ, ddcc.FIELD_P]
    host, snap = state["host"], state["snapshot"]
    for k, field in enumerate(ids):
        _lib.ddcc3d_read(sim.h, field, host[k].numpy())
    if snap is not host:
        snap.copy_(host)
    n = case["phases"] - 1
    return dict(C=snap[:n], u=snap[n:n + 3], P=snap[n + 3])


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------

def work(case):
    """Bytes: per step the state read and written once and the static fields
    read once; the results written once.  Operations per node and step as
    counted in the equations of ``_Model2D`` / ``_Model3D`` (additions,
    multiplications and divisions, no halo computed twice)."""
    N, T, e = case["phases"], case["steps"], 8 if case["f64"] else 4
    static = 1 + (N - 1 if case["field"] or case.get("scene") == "channel" else 0)
    if case["kind"] == "step3d":
        n = case["nx"] * case["ny"] * case["nz"]
        planes = 7 * (N - 1) + 15 + 3 * N + 7
        out = (N + 3) * n * (8 + (0 if case["f64"] else 4))
        return dict(bytes=n * e * (2 * planes + static) * T + out, flops=n * T * {2: 1150, 3: 1550, 4: 2050}[N])
    n = case["nx"] * case["ny"]
    planes = 11 * N + 3
    flops = {2: 520, 3: 850, 4: 1250}[N]
    step = n * e * (2 * planes + static)
    if case["kind"] == "monitor2d":
        return dict(bytes=step * T + n * 8 * (2 * N + 4), flops=n * flops * T)
    if case["kind"] == "step2d":
        return dict(bytes=step * T + 2 * n * e * planes, flops=n * flops * T)
    # forward sweep; per reverse step the state of that step formed again and
    # read with the adjoint state, which is written back, and the gradient
    # planes (64-bit sums) read and written
    reverse = step + n * e * (3 * planes + static) + n * 16 * N
    return dict(bytes=T * (step + reverse) + n * (8 + 2 * e) * N, flops=n * T * flops * 5)


# ----------------------------------------------------------------------------
# the same results in 64 bits
# ----------------------------------------------------------------------------

class _Stencil:
    """Neighbour values on a grid: periodic wrap or mirror about an outer wall."""

    def __init__(self, shape, periodic, device):
        self.index = []
        for n, per in zip(shape, periodic):
            i = torch.arange(-1, n + 1, device=device)
            self.index.append(i % n if per else torch.clamp(i, 0, n - 1))
        self.shape = shape

    def padded(self, f):
        k = len(self.shape)
        for a, idx in enumerate(self.index):
            f = f.index_select(f.dim() - k + a, idx)
        return f

    def shifted(self, fp, c):
        """Values at x + c (c in x, y[, z] order) of a padded field."""
        sl = [Ellipsis] + [slice(1 + d, 1 + d + n) for d, n in zip(reversed(c), self.shape)]
        return fp[tuple(sl)]


class _Model:
    """What the two- and the three-dimensional step share: gradients, chemical
    potentials, mobility flux and the velocity / pressure solve."""

    def __init__(self, prm, psi, cos, walls, shape, periodic):
        self.p, self.N, self.dev = prm, prm["nphase"], psi.device
        self.shape, self.periodic, self.dim = shape, periodic, len(shape)
        self.st = _Stencil(shape, periodic, self.dev)
        self.psi = psi
        self.psi_pad = self.st.padded(psi)
        self.cs2 = prm["d0"]
        self.gpsi = self.grad(psi)
        if walls is None:
            g2 = sum(g * g for g in self.gpsi)
            flat = g2 <= 1e-12          # |grad psi| counts as having no slope there
            self.agp = torch.where(flat, torch.sqrt(g2.detach()), torch.sqrt(torch.where(flat, 1.0, g2)))
            self.cos = cos
        else:                           # wetting strengths summed over the solids
            self.agp = torch.ones_like(psi)
            self.cos = sum(c * torch.sqrt(sum(g * g for g in self.grad(pk))) for pk, c in walls)
        self.sig = torch.tensor(prm["sigma"], dtype=torch.float64, device=self.dev)

    def vec(self, values):
        return torch.tensor(list(values), dtype=torch.float64, device=self.dev)

    def col(self, values, extra=0):
        return self.vec(values).reshape((-1,) + (1,) * (self.dim + extra))

    def grad(self, f):
        """sum_p w_p c_p f(x + c_p) / cs2 on the flow lattice."""
        fp = self.st.padded(f)
        out = [0.0] * self.dim
        for c, w in zip(self.c, self.w):
            if not any(c):
                continue
            v = (w / self.cs2) * self.st.shifted(fp, c)
            out = [o + v if d > 0 else o - v if d < 0 else o for o, d in zip(out, c)]
        return out

    def chem_pot(self, C):
        """mu_i of all phases from the fractions of all phases (Eq. 2.14)."""
        Cp = self.st.padded(C)
        lap = 0.0
        for c, w in zip(self.c, self.w):
            if any(c):
                lap = lap + (w / self.cs2) * (self.psi + self.st.shifted(self.psi_pad, c)) * \
                    (self.st.shifted(Cp, c) - C)
        gp = lambda v: 2.0 * v * (v - 1.0) * (2.0 * v - 1.0)  # noqa: E731
        N, eps = self.N, self.p["width"]
        mu = []
        wet = []
        aj = [self.p["sigma"][j][N - 1] * self.cos[j] for j in range(N - 1)] + [torch.zeros_like(self.psi)]
        for j in range(N):
            s = 0.0
            for q in range(N):
                if q != j:
                    s = s + (aj[j] - aj[q]) / self.p["sigma"][j][q] * C[q]
            wet.append(C[j] * s)
        for i in range(N):
            m = 0.0
            for j in range(N):
                if j == i:
                    continue
                s = self.p["sigma"][i][j]
                m = m + (6.0 * s / eps) * self.psi * (gp(C[i]) - gp(C[i] + C[j])) + 0.75 * eps * s * lap[j] \
                    + 3.0 * s * self.agp * wet[j]
            mu.append(m / self.psi)
        return torch.stack(mu)

    def macro(self, f, g, lag_a, lag_pm):
        """Everything the update needs from the current state: fractions,
        potentials, gradients, force and the joint velocity / pressure solve."""
        p, N, psi, d = self.p, self.N, self.psi, self.dim
        m = {}
        psiC = f.sum(1)
        C = psiC / psi
        C = torch.cat([C, (1.0 - C.sum(0))[None]])
        mu = self.chem_pot(C)
        gC, gmu = self.grad(C), self.grad(mu)
        rho_i = self.col(p["rho"])
        rho, nu = (rho_i * C).sum(0), (self.col(p["nu"]) * C).sum(0)
        grho = [(rho_i * gC[a]).sum(0) for a in range(d)]
        gpr = self.grad(psi * rho)
        S = C.sum(0)
        G = [(C * gmu[a]).sum(0) for a in range(d)]
        Q = [C * (S * gmu[a] - G[a]) for a in range(d)]           # sum_j M_ij grad mu_j / m0
        mC = [-p["m0"] * (rho_i * Q[a]).sum(0) for a in range(d)]
        F0 = [(psi * mu * gC[a]).sum(0) + psi * rho * p["body_force"][a] for a in range(d)]
        ga = [self.grad(a) for a in lag_a]
        if d == 2:
            F0[0] = F0[0] + ga[0][1]
            F0[1] = F0[1] - ga[0][0]
        else:
            F0[0] = F0[0] + ga[0][1] - ga[2][2]
            F0[1] = F0[1] + ga[1][2] - ga[0][0]
            F0[2] = F0[2] + ga[2][0] - ga[1][1]
        J = [sum(c[a] * g[k] for k, c in enumerate(self.c) if c[a]) for a in range(d)]
        sum_g = g[1:].sum(0)
        cs2, d0, w0 = self.cs2, p["d0"], self.w[0]
        s21 = 1.0 / (nu * 2.0 / (1.0 - cs2) + 0.5)
        s22 = 1.0 / (nu / cs2 + 0.5)
        K = 1.0 - d0 if d == 2 else 1.0 - 2.0 * d0
        H = K * (1.0 - 2.0 * d0) if d == 2 else K * (3.0 - 7.0 * d0) / 2.0
        H = H * (s21 - 2.0) / s21
        s0 = p["s_g"][0]
        A_P = 0.5 + K * (1.0 - d0) * (2.0 - s0) / (2.0 * s0)
        gam, cP = K / 2.0 - w0 / (1.0 - cs2), cs2 / (1.0 - w0)
        damp = (1.0 - psi) / p["eps0"] ** 3
        den = psi * rho + 0.5 * damp
        u0 = [(J[a] + 0.5 * F0[a]) / den for a in range(d)]
        e = [0.5 * self.gpsi[a] / den for a in range(d)]
        b = [A_P * psi * grho[a] + gam * psi * mC[a] + H * gpr[a] for a in range(d)]
        dot = lambda u, v: sum(u[a] * v[a] for a in range(d))  # noqa: E731
        q = gam * psi * rho
        qa = cP * q * dot(e, e)
        qb = cP * (dot(b, e) + 2.0 * q * dot(u0, e)) - psi
        qc = cP * (sum_g - 0.5 * K * lag_pm + dot(b, u0) + q * dot(u0, u0))
        root = torch.sqrt(torch.clamp(qb * qb - 4.0 * qa * qc, min=0.0))
        P = -2.0 * qc / torch.where(qb < 0.0, qb - root, qb + root)
        u = [u0[a] + P * e[a] for a in range(d)]
        F = [F0[a] + P * self.gpsi[a] - damp * u[a] for a in range(d)]
        m.update(C=C, mu=mu, rho=rho, u=u, P=P, F=F, Q=Q, mC=mC, gmu=gmu, grho=grho, gpr=gpr, s21=s21, s22=s22,
                 psiC=psiC)
        return m

    def phase_equilibrium0(self, C0):
        """Phase populations of the initial state (u = 0)."""
        C = torch.cat([C0, (1.0 - C0.sum(0))[None]])
        emu = self.col(self.p["eta"]) * self.psi * self.chem_pot(C)[:-1]
        w = self.col(self.wf, 0)
        f = w[None] * emu[:, None]
        rest = (self.wf[0] - 1.0) * emu + self.psi * C0
        return torch.cat([rest[:, None], f[:, 1:]], 1)

    def stream(self, out, vel):
        """Push to x + c, or back in the opposite direction off an outer wall."""
        k = self.dim
        opp = [vel.index(tuple(-v for v in c)) for c in vel]
        new = []
        for q, c in enumerate(vel):
            # population q arrives from x - c, or from the node's own opposite
            src = out.select(out.dim() - k - 1, q)
            moved = src
            for a in range(k):
                if c[k - 1 - a]:
                    moved = torch.roll(moved, c[k - 1 - a], moved.dim() - k + a)
            outside = None
            for a in range(k):
                step, per, n = c[k - 1 - a], self.periodic[a], self.shape[a]
                if step and not per:
                    i = torch.arange(n, device=self.dev)
                    edge = (i == 0) if step > 0 else (i == n - 1)
                    edge = edge.reshape([n if b == a else 1 for b in range(k)])
                    outside = edge if outside is None else outside | edge
            if outside is not None:
                moved = torch.where(outside, out.select(out.dim() - k - 1, opp[q]), moved)
            new.append(moved)
        return torch.stack(new, out.dim() - k - 1)

    def relax(self, v, H, w, k):
        """v_p - w_p sum_k h_k(c_p) k_k."""
        B = torch.einsum("kp,k...->p...", H, k)
        return v - self.col(w) * B


class _Model2D(_Model):
    c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]

    def __init__(self, prm, psi, cos, walls=None):
        d0 = prm["d0"]
        w1 = {0: 1.0 - d0, 1: d0 / 2.0, -1: d0 / 2.0}
        self.w = self.wf = [w1[a] * w1[b] for a, b in self.c]
        super().__init__(prm, psi, cos, walls, (prm["ny"], prm["nx"]), (prm["periodic_y"], prm["periodic_x"]))
        h = lambda k, c: (1.0, c, c * c - d0)[k]  # noqa: E731
        self.order = [(0, 0), (1, 0), (0, 1), (2, 0), (0, 2), (1, 1), (2, 1), (1, 2), (2, 2)]
        self.H = self.vec([h(a, x) * h(b, y) for a, b in self.order for x, y in self.c]).reshape(9, 9)
        n = (1.0, d0, d0 * (1.0 - d0))
        self.norm = [n[a] * n[b] for a, b in self.order]

    def start(self, C0):
        N = self.N
        zero = lambda k: torch.zeros((k,) + self.shape, dtype=torch.float64, device=self.dev)  # noqa: E731
        return self.phase_equilibrium0(C0), zero(9), zero(2 * N + 3)

    def fields(self, f, g, lag):
        return self.macro(f, g, [lag[0]], lag[2 * self.N + 2])

    def step(self, f, g, lag):
        p, N, psi, cs2, nrm = self.p, self.N, self.psi, self.cs2, self.norm
        m = self.fields(f, g, lag)
        ux, uy = m["u"]
        gpx, gpy = self.gpsi
        new_f, lag_cu = [], []
        for i in range(N - 1):
            M = torch.einsum("kp,p...->k...", self.H, f[i])
            eta = p["eta"][i]
            s1 = 1.0 / (p["m0"] / (eta * cs2) + 0.5)
            s0, s21, s22, s3, s4 = p["s_f"]
            rate = [s0, s1, s1, s21, s21, s22, s3, s3, s4]
            pc = (m["psiC"][i] * ux, m["psiC"][i] * uy)
            V = []
            for a in range(2):
                S = psi * (m["Q"][a][i] - m["gmu"][a][i])
                V.append(pc[a] - lag[1 + 2 * i + a] + cs2 * eta * (m["mu"][i] * self.gpsi[a] - S))
            X = m["psiC"][i] - eta * psi * m["mu"][i]
            k = [torch.zeros_like(psi)]
            k += [rate[1 + a] / nrm[1 + a] * (M[1 + a] - pc[a] + 0.5 * V[a]) - V[a] / nrm[1 + a] for a in range(2)]
            k += [rate[b] / nrm[b] * (M[b] + cs2 * X) for b in (3, 4)]
            k += [rate[b] / nrm[b] * M[b] for b in (5, 6, 7)]
            k.append(rate[8] / nrm[8] * (M[8] - cs2 * cs2 * X))
            new_f.append(self.relax(f[i], self.H, self.w, torch.stack(k)))
            lag_cu += list(pc)
        rho, (mx, my) = m["rho"], m["mC"]
        pr = psi * rho
        T = (psi * mx * ux, psi * my * uy, 0.5 * psi * (mx * uy + ux * my))
        A = (pr * ux * ux + T[0], pr * uy * uy + T[1], pr * ux * uy + T[2])
        gx, gy = m["gpr"]
        ug = (1.0 - 3.0 * cs2) * (ux * gx + uy * gy)
        D = (T[0] - lag[2 * N - 1] + 2.0 * cs2 * ux * gx + ug, T[1] - lag[2 * N] + 2.0 * cs2 * uy * gy + ug,
             T[2] - lag[2 * N + 1] + cs2 * (ux * gy + gx * uy))
        a0 = psi * (ux * m["grho"][0] + uy * m["grho"][1])
        pP = psi * m["P"]
        M = torch.einsum("kp,p...->k...", self.H, g)
        s0, s1, s3, s4 = p["s_g"]
        F, s21, s22 = m["F"], m["s21"], m["s22"]
        k = [s0 * (M[0] + 0.5 * a0) - a0]
        k += [(s1 * (M[1 + a] - pr * m["u"][a] + 0.5 * F[a]) - F[a]) / nrm[1 + a] for a in range(2)]
        k += [(s21 * (M[3 + a] - pP - A[a] + 0.5 * D[a]) - D[a]) / nrm[3 + a] for a in range(2)]
        k.append((s22 * (M[5] - A[2] + 0.5 * D[2]) - D[2]) / nrm[5])
        k += [s3 / nrm[6] * M[6], s3 / nrm[7] * M[7], s4 / nrm[8] * (M[8] + cs2 * pP)]
        new_g = self.relax(g, self.H, self.w, torch.stack(k))
        pm = psi * (rho * (ux * ux + uy * uy) + mx * ux + my * uy)
        new_lag = torch.stack([0.5 * psi * (mx * uy - ux * my)] + lag_cu + list(T) + [pm])
        return self.stream(torch.stack(new_f), self.c), self.stream(new_g, self.c), new_lag

    def open_ends(self, f, g, lag, u_in, C_in):
        """Equilibrium at the inflow and outflow columns of a streamed state."""
        p, N, cs2, nx = self.p, self.N, self.cs2, self.p["nx"]
        K, cP = 1.0 - p["d0"], cs2 / (1.0 - self.w[0])
        w = self.vec(self.w)[:, None]
        cx = self.vec(c[0] for c in self.c)[:, None]
        rest = torch.zeros(9, 1, dtype=torch.float64, device=self.dev)
        rest[0] = 1.0
        for b, n in ((0, 1), (nx - 1, nx - 2)):
            psib, psin = self.psi[:, b], self.psi[:, n]
            C = C_in if b == 0 else f[:, :, :, n].sum(1) / psin
            rho = (self.vec(p["rho"][:N - 1])[:, None] * C).sum(0) + p["rho"][N - 1] * (1.0 - C.sum(0))
            pP = psib * cP * (g[1:, :, n].sum(0) - 0.5 * K * lag[2 * N + 2, :, n]) / psin
            pC = psib * C
            f[:, :, :, b] = rest * pC[:, None] + w * cx * (pC * u_in / cs2)[:, None] * (1.0 - rest)
            pru = psib * rho * u_in
            g[:, :, b] = (w - rest) * pP / cs2 + w * (cx * pru / cs2 + pru * u_in * (cx * cx - cs2) /
                                                      (cs2 - cs2 * cs2))
            lag[:, :, b] = 0.0
            lag[1:2 * N - 1:2, :, b] = pC * u_in
            lag[2 * N + 2, :, b] = pru * u_in
        return f, g, lag


class _Model3D(_Model):
    c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + \
        [(1 - 2 * (b & 1), 1 - (b & 2), 1 - (b & 4) // 2) for b in range(8)]

    def __init__(self, prm, psi, cos):
        d0 = prm["d0"]
        w0 = 1.0 - 3.0 * d0 + 2.0 * d0 * d0
        self.w = [w0] + [(d0 - d0 * d0) / 2.0] * 6 + [d0 * d0 / 8.0] * 8
        self.wf = [1.0 - 3.0 * d0] + [d0 / 2.0] * 6
        super().__init__(prm, psi, cos, None, (prm["nz"], prm["ny"], prm["nx"]), (1, 1, 1))
        rows = []
        for x, y, z in self.c:
            rows.append([1.0, x, y, z, x * x - d0, y * y - d0, z * z - d0, x * y, y * z, z * x, x * (y * y - d0),
                         y * (z * z - d0), z * (x * x - d0), x * y * z,
                         (x * y * z) ** 2 - d0 * (x * x + y * y + z * z) + 2.0 * d0 * d0])
        self.H = self.vec(v for k in range(15) for v in (r[k] for r in rows)).reshape(15, 15)
        self.norm = [1.0] + [d0] * 3 + [d0 * (1.0 - d0)] * 3 + [d0 * d0] * 3 + [d0 * d0 * (1.0 - d0)] * 3 + \
            [d0 * d0, d0 * d0 * w0]

    def start(self, C0):
        zero = lambda k: torch.zeros((k,) + self.shape, dtype=torch.float64, device=self.dev)  # noqa: E731
        return self.phase_equilibrium0(C0), zero(15), zero(3 * self.N + 7)

    def fields(self, f, g, lag):
        return self.macro(f, g, [lag[0], lag[1], lag[2]], lag[3 * self.N + 6])

    def step(self, f, g, lag):
        p, N, psi, cs2, nrm = self.p, self.N, self.psi, self.cs2, self.norm
        m = self.fields(f, g, lag)
        u, mC, gpr = m["u"], m["mC"], m["gpr"]
        w1 = self.wf[1]
        new_f, lag_cu = [], []
        for i in range(N - 1):
            eta = p["eta"][i]
            s1 = 1.0 / (p["m0"] / (eta * cs2) + 0.5)
            epm = eta * psi * m["mu"][i]
            out, total = [None] * 7, 0.0
            for a in range(3):
                S = psi * (m["Q"][a][i] - m["gmu"][a][i])
                cu = m["psiC"][i] * u[a]
                V = cu - lag[3 + 3 * i + a] + cs2 * eta * (m["mu"][i] * self.gpsi[a] - S)
                fp, fm = f[i, 1 + 2 * a], f[i, 2 + 2 * a]
                odd = s1 * (fp - fm - cu + 0.5 * V)
                even = p["s_f"][1] * (fp + fm - cs2 * epm)
                out[1 + 2 * a] = fp - 0.5 * (even + odd) + w1 * V / cs2
                out[2 + 2 * a] = fm - 0.5 * (even - odd) - w1 * V / cs2
                total = total + even
                lag_cu.append(cu)
            out[0] = f[i, 0] + total
            new_f.append(torch.stack(out))
        rho = m["rho"]
        pr = psi * rho
        nxt = (1, 2, 0)
        T = [psi * mC[a] * u[a] for a in range(3)] + \
            [0.5 * psi * (mC[a] * u[b] + u[a] * mC[b]) for a, b in enumerate(nxt)]
        A = [pr * u[a] * u[a] + T[a] for a in range(3)] + [pr * u[a] * u[b] + T[3 + a] for a, b in enumerate(nxt)]
        ug = (1.0 - 3.0 * cs2) * sum(u[a] * gpr[a] for a in range(3))
        old = lag[3 * N:3 * N + 6]
        D = [T[a] - old[a] + 2.0 * cs2 * u[a] * gpr[a] + ug for a in range(3)] + \
            [T[3 + a] - old[3 + a] + cs2 * (u[a] * gpr[b] + gpr[a] * u[b]) for a, b in enumerate(nxt)]
        a0 = psi * sum(u[a] * m["grho"][a] for a in range(3))
        pP = psi * m["P"]
        M = torch.einsum("kp,p...->k...", self.H, g)
        s0, s1, s3, s4 = p["s_g"]
        F, s21, s22 = m["F"], m["s21"], m["s22"]
        k = [s0 * (M[0] + 0.5 * a0) - a0]
        k += [(s1 * (M[1 + a] - pr * u[a] + 0.5 * F[a]) - F[a]) / nrm[1] for a in range(3)]
        k += [(s21 * (M[4 + a] - pP - A[a] + 0.5 * D[a]) - D[a]) / nrm[4] for a in range(3)]
        k += [(s22 * (M[7 + a] - A[3 + a] + 0.5 * D[3 + a]) - D[3 + a]) / nrm[7] for a in range(3)]
        k += [s3 / nrm[b] * M[b] for b in (10, 11, 12, 13)]
        k.append(s4 / nrm[14] * (M[14] + 2.0 * cs2 * pP))
        new_g = self.relax(g, self.H, self.w, torch.stack(k))
        a_new = [0.5 * psi * (mC[a] * u[b] - u[a] * mC[b]) for a, b in enumerate(nxt)]
        pm = psi * sum(rho * u[a] * u[a] + mC[a] * u[a] for a in range(3))
        new_lag = torch.stack(a_new + lag_cu + T + [pm])
        vel = self.c
        return self.stream(torch.stack(new_f), vel[:7]), self.stream(new_g, vel), new_lag


def exact(case, seed):
    dev = _device()
    t = lambda a: None if a is None else torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64,  # noqa: E731
                                                         device=dev)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    inp = _inputs3d(case, seed) if case["kind"] == "step3d" else _inputs2d(case, seed)
    prm = inp["params"]
    psi, C0 = t(inp["psi"]), t(inp["C0"])
    one = (1,) * psi.dim()
    cos = t(inp["cos_field"]) if inp["cos_field"] is not None else None
    if cos is None and inp["cos"] is not None:
        cos = t(inp["cos"]).reshape((-1,) + one).expand((-1,) + tuple(psi.shape))
    with torch.no_grad():
        if case["kind"] == "step3d":
            model = _Model3D(prm, psi, cos)
            s = model.start(C0)
            for _ in range(case["steps"]):
                s = model.step(*s)
            m = model.fields(*s)
            return dict(C=m["C"][:-1], u=torch.stack(m["u"]), P=m["P"])
        walls = inp["walls"]
        if walls is not None:
            walls = [(t(p), t(c).reshape((-1,) + one)) for p, c in walls]
        model = _Model2D(prm, psi, cos, walls)
        s = model.start(C0)
        ends = None if inp["open_x"] is None else [t(v) for v in inp["open_x"]]
        for _ in range(case["steps"]):
            s = model.step(*s)
            if ends is not None:
                s = model.open_ends(*s, *ends)
        f, g, lag = s
        if case["kind"] == "monitor2d":
            m = model.fields(*s)
            return dict(C=m["C"], rho=m["rho"], ux=m["u"][0], uy=m["u"][1], P=m["P"], mu=m["mu"],
                        mass=f.sum((1, 2, 3)))
        return dict(f=f.reshape((-1,) + tuple(psi.shape)), g=g, lag=lag)


def _exact_adjoint(case, seed):
    """Gradients by automatic differentiation of the 64-bit step, one
    checkpointed segment at a time."""
    dev = _device()
    real = torch.float64 if case["f64"] else torch.float32
    inp = _inputs2d(case, seed)
    leaf = lambda a: torch.tensor(a, dtype=real, device=dev).double().requires_grad_(True)  # noqa: E731
    cos, psi = leaf(inp["cos_field"]), leaf(inp["psi"])
    C0 = torch.tensor(inp["C0"], dtype=torch.float64, device=dev)
    T, seg = case["steps"], 5
    with torch.no_grad():
        model = _Model2D(inp["params"], psi, cos)
        s = model.start(C0)
        heads = []
        for n in range(T):
            if n % seg == 0:
                heads.append(s)
            s = model.step(*s)
    x = torch.arange(case["nx"], dtype=torch.float64, device=dev)
    m = s[0][0].sum(0)
    J = (x * m).sum() / m.sum()
    bar_f = torch.zeros_like(s[0])
    bar_f[0] = ((x - J) / m.sum()).expand(9, case["ny"], case["nx"])
    bar = [bar_f, torch.zeros_like(s[1]), torch.zeros_like(s[2])]
    gc, gp = torch.zeros_like(cos), torch.zeros_like(psi)
    for k in range(len(heads) - 1, -1, -1):
        state = [v.detach().requires_grad_(True) for v in heads[k]]
        model = _Model2D(inp["params"], psi, cos)
        s = state
        for _ in range(min(seg, T - k * seg)):
            s = model.step(*s)
        got = torch.autograd.grad(s, state + [cos, psi], bar, allow_unused=True)
        bar = [torch.zeros_like(v) if b is None else b for v, b in zip(state, got[:3])]
        gc, gp = gc + got[3], gp + got[4]
    f0 = _Model2D(inp["params"], psi, cos).start(C0)[0]
    got = torch.autograd.grad(f0, [cos, psi], bar[0])
    return dict(J=J, dJ_dcos=gc + got[0], dJ_dpsi=gp + got[1])
