"""Performance cases of the EREM library: the calls its users make, over the
sizes, precisions and options they make them with.

Every case goes through the package's public entry points (``Context``,
``Ensemble``, ``MisfitModel``/``misfit``).  Two families of fields, both of
the shapes of ``workloads``:

* ``layers``: a 3D reservoir of horizontal layers with x-aligned channels of
  permeability 1e4.  ln K depends on (y, z) only, so the steady pressure is
  the linear ramp from head_left to head_right.
* ``gauss``: a Gaussian log-permeability field (2D or 3D), whose pressure the
  program has solved with the library before it steps.

``exact`` gives the same results in FP64 torch on its own: the heat operator
and the pressure matrix assembled from the fields, the pressure by Jacobi CG,
and the exponential integrator as the exact solution of the linear(ized) heat
equation over the run (Taylor steps of the semi-discrete system), which the
real Leja and Krylov forms approximate to their tolerance of 1e-6.
"""
import math

import torch

import paper_1209_5553_gb300 as E
from paper_1209_5553_gb300.autograd import MisfitModel, misfit

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one FP64 step of the 64 x 64 workload (interactive
        # use and parameter sweeps; launches and waits decide)
        dict(name="step2d_64_fp64", op="steps", field="gauss", nx=64, ny=64, nz=1, precision="fp64",
             steps=1, dt=0.05, sigma=1.0, ell=0.1),
        # a ragged 2D grid in the default precision, a short run
        dict(name="run2d_517x389_fp64", op="steps", field="gauss", nx=517, ny=389, nz=1,
             precision="fp64", steps=3, dt=0.02, sigma=1.5, ell=0.1),
        # the headline workload: 256^3 layered reservoir, FP32-bulk, a run of steps
        dict(name="run3d_256_fp32", op="steps", field="layers", nx=256, ny=256, nz=256,
             precision="fp32_bulk", steps=4, dt=8.0 / 256),
        # a ragged heterogeneous 3D grid in FP64
        dict(name="run3d_101x77x59_fp64", op="steps", field="gauss", nx=101, ny=77, nz=59,
             precision="fp64", steps=2, dt=0.02, sigma=1.0, ell=0.15),
        # new fields, then one action of tau phi_1(tau J) on a vector (a caller
        # with its own time stepping): assembly and one interpolation
        dict(name="assemble_phi1_192_fp32", op="phi1", field="layers", nx=192, ny=192, nz=192,
             precision="fp32_bulk", steps=1, dt=8.0 / 192),
        # a steady pressure from the ramp guess, 3D heterogeneous
        dict(name="pressure3d_128", op="pressure", field="gauss", nx=128, ny=128, nz=128,
             precision="fp64", steps=1, dt=0.01, sigma=2.0, ell=0.05),
        # the coupled pressure/temperature step with T-dependent fluid laws
        dict(name="coupled2d_1024_fp32", op="coupled", field="gauss", nx=1024, ny=1024, nz=1,
             precision="fp32_bulk", steps=1, dt=0.005, sigma=2.0, ell=0.02),
        # the Rosenbrock alternative on the coupled problem (FP64, implicit)
        dict(name="ros2_512", op="ros2", field="gauss", nx=512, ny=512, nz=1, precision="fp64",
             steps=1, dt=0.005, sigma=2.0, ell=0.02),
        # time-dependent inflow temperature: phi_1 and phi_2 parts
        dict(name="forced3d_128_fp32", op="forced", field="layers", nx=128, ny=128, nz=128,
             precision="fp32_bulk", steps=2, dt=8.0 / 128),
        # the Krylov form of the same step
        dict(name="krylov3d_112", op="krylov", field="layers", nx=112, ny=112, nz=112,
             precision="fp64", steps=1, dt=8.0 / 112),
        # an ensemble of independent 2D members of mixed sizes
        dict(name="ensemble_24_fp32", op="ensemble", field="gauss", nx=64, ny=320, nz=1,
             precision="fp32_bulk", steps=4, dt=0.05, sigma=1.5, ell=0.1, members=24),
        # one gradient of the misfit (forward and backward) by the adjoint
        dict(name="gradient3d_64_fp32", op="gradient", field="layers", nx=64, ny=64, nz=64,
             precision="fp32_bulk", steps=8, dt=4.0 / 64),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["steps2", "steps3", "steps3", "phi1", "pressure", "coupled", "rosm", "forced", "krylov",
                     "ensemble", "gradient"])
    prec = rng.choice(["fp64", "fp32_bulk"])
    if op == "steps2":
        nx, ny = _size(rng, 24, 1200), _size(rng, 24, 1200)
        return dict(op="steps", field="gauss", nx=nx, ny=ny, nz=1, precision=prec, steps=rng.randint(1, 4),
                    dt=8.0 / max(nx, ny, 160), sigma=round(rng.uniform(0.5, 2.0), 3), ell=0.1)
    if op == "steps3":
        if rng.random() < 0.5:
            nx, ny, nz = (_size(rng, 16, 256) for _ in range(3))
            return dict(op="steps", field="layers", nx=nx, ny=ny, nz=nz, precision=prec,
                        steps=rng.randint(1, 3), dt=8.0 / max(nx, ny, nz))
        nx, ny, nz = (_size(rng, 12, 128) for _ in range(3))
        return dict(op="steps", field="gauss", nx=nx, ny=ny, nz=nz, precision=prec, steps=rng.randint(1, 3),
                    dt=2.0 / max(nx, ny, nz), sigma=round(rng.uniform(0.5, 1.5), 3), ell=0.15)
    if op in ("phi1", "forced", "krylov"):
        hi = 200 if op == "phi1" else 112
        nx, ny, nz = (_size(rng, 16, hi) for _ in range(3))
        return dict(op=op, field="layers", nx=nx, ny=ny, nz=nz,
                    precision="fp64" if op == "krylov" else prec, steps=1, dt=8.0 / max(nx, ny, nz))
    if op == "pressure":
        nz = rng.choice([1, _size(rng, 8, 96)])
        hi = 900 if nz == 1 else 110
        nx, ny = _size(rng, 16, hi), _size(rng, 16, hi)
        return dict(op="pressure", field="gauss", nx=nx, ny=ny, nz=nz, precision="fp64", steps=1, dt=0.01,
                    sigma=round(rng.uniform(0.5, 2.0), 3), ell=0.05)
    if op in ("coupled", "rosm"):
        nx, ny = _size(rng, 32, 640), _size(rng, 32, 640)
        return dict(op=rng.choice(["ros2", "ros3p"]) if op == "rosm" else "coupled", field="gauss",
                    nx=nx, ny=ny, nz=1, precision="fp64" if op == "rosm" else prec, steps=1, dt=0.005,
                    sigma=round(rng.uniform(0.5, 2.0), 3), ell=0.05)
    if op == "ensemble":
        return dict(op="ensemble", field="gauss", nx=48, ny=_size(rng, 100, 320), nz=1, precision=prec,
                    steps=rng.randint(1, 4), dt=0.05, sigma=round(rng.uniform(0.5, 2.0), 3), ell=0.1,
                    members=rng.randint(4, 20))
    nx, ny, nz = (_size(rng, 16, 64) for _ in range(3))
    return dict(op="gradient", field="layers", nx=nx, ny=ny, nz=nz, precision=prec, steps=rng.randint(2, 8),
                dt=4.0 / max(nx, ny, nz))


# ---------------------------------------------------------------------------
# fields
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _gauss(shape, ell, sigma, gen):
    """Zero-mean Gaussian field of standard deviation sigma and correlation
    length ell on the unit cube (periodic), by spectral synthesis."""
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, device=DEV, dtype=F64))
    k2 = torch.zeros((), device=DEV, dtype=F64)
    for d, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device=DEV, dtype=F64) if d == len(shape) - 1 else \
            torch.fft.fftfreq(n, device=DEV, dtype=F64)
        s = [1] * len(shape)
        s[d] = -1
        k2 = k2 + (k * n).reshape(s) ** 2
    x = torch.fft.irfftn(f * torch.exp(-(math.pi * ell) ** 2 * k2), s=shape)
    x = x - x.mean()
    return (x * (sigma / x.std())).reshape(-1)


def _centres(n):
    return (torch.arange(n, device=DEV, dtype=F64) + 0.5) / n


class Fields:
    """What a user's program holds: the fields and constants of one problem."""

    def __init__(self, c, seed, nx=None, ny=None):
        self.nx, self.ny, self.nz = nx or c["nx"], ny or c["ny"], c["nz"]
        nx, ny, nz = self.nx, self.ny, self.nz
        self.dim = 3 if nz > 1 else 2
        self.N = nx * ny * nz
        self.shape = (nz, ny, nx)
        self.dt = c["dt"]
        g = _gen(seed)
        x = _centres(nx).expand(self.shape)
        coupled = c["op"] in ("coupled", "ros2", "ros3p")
        if c["field"] == "layers":
            m = torch.randn((min(16, nz),), generator=g, device=DEV, dtype=F64)
            yz = m[torch.arange(nz, device=DEV) * len(m) // nz].reshape(nz, 1).repeat(1, ny)
            wy, wz = max(1, ny // 32), max(1, nz // 32)
            for _ in range(8):  # x-aligned channels
                r = torch.rand((2,), generator=g, device=DEV, dtype=F64).tolist()
                j, k = int(r[0] * (ny // wy)) * wy, int(r[1] * (nz // wz)) * wz
                yz[k:k + wz, j:j + wy] = math.log(1e4)
            self.lnk = yz.reshape(nz, ny, 1).expand(self.shape).reshape(-1).contiguous()
            # the largest face speed is 1 (K = 1e4 in the channels), Pe = 1e3
            self.phys = E.Physics(1e3, 1e3, 1e-4, 0.0, 80.0, 0)
            self.p = (1e-4 * (1.0 - x)).reshape(-1).contiguous()
            self.phi = torch.full((self.N,), 0.2, device=DEV, dtype=F64)
            self.lam = torch.full((self.N,), 1.0, device=DEV, dtype=F64)
        else:
            sh = self.shape if self.dim == 3 else self.shape[1:]
            self.lnk = _gauss(sh, c["ell"], c["sigma"], g)
            # geometric mean permeability 1 and a head drop of 1: Pe = 50
            self.phys = E.Physics(100.0, 100.0, 1.0, 0.0, 80.0, 1 if coupled else 0)
            self.p = (1.0 - x).reshape(-1).contiguous()   # the guess a solve starts from
            if self.dim == 3:  # heterogeneous rock
                self.phi = 0.1 + 0.25 * torch.rand((self.N,), generator=g, device=DEV, dtype=F64)
                self.lam = 1.0 + 2.0 * torch.rand((self.N,), generator=g, device=DEV, dtype=F64)
            else:
                self.phi = torch.full((self.N,), 0.2, device=DEV, dtype=F64)
                self.lam = torch.full((self.N,), 2.0, device=DEV, dtype=F64)
        # initial temperature: 20 with a geothermal gradient in depth, a smooth
        # disturbance, and (coupled) a front that has entered from x = 0
        depth = _centres(nz).reshape(-1, 1, 1) if nz > 1 else _centres(ny).reshape(1, -1, 1)
        a = torch.rand((4,), generator=g, device=DEV, dtype=F64)
        y = _centres(ny).reshape(1, -1, 1)
        T = 20.0 + 15.0 * depth + 3.0 * torch.sin(6.28 * (a[0] + (1.0 + a[1]) * x)) * torch.cos(6.28 * (a[2] + y))
        if coupled:
            T = 24.0 + 0.2 * (T - 24.0) + 50.0 * torch.exp(-(x / (0.08 + 0.02 * torch.sin(6.28 * (a[3] + y)))) ** 2)
        self.T0 = T.expand(self.shape).reshape(-1).contiguous()


def _members(c, seed):
    """Grid sizes of an ensemble: n x n, spread over [nx, ny] (the same for every
    seed: the sizes belong to the case)."""
    n, lo, hi = c["members"], c["nx"], c["ny"]
    return [(lo + (hi - lo) * ((7 * e) % n) // max(1, n - 1), 1000 * seed + e) for e in range(n)]


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
PTOL = 1e-12      # steady pressures solved before a run
FORCED = (72.0, -160.0)   # inflow temperature at t_n and its rate


class State:
    pass


def prepare(case, seed):
    c, s = case, State()
    s.case = c
    if c["op"] == "ensemble":
        s.f = [Fields(c, sd, n, n) for n, sd in _members(c, seed)]
        s.ens = E.Ensemble([(f.nx, f.ny, f.phys) for f in s.f], precision=c["precision"])
        for e, f in enumerate(s.f):
            with E.Context(2, f.nx, f.ny, physics=f.phys) as ctx:
                ctx.pressure_solve(f.lnk, None, f.p, tol=PTOL)
            s.ens.set_member(e, f.T0, f.p, f.lnk, f.phi, f.lam, f.dt)
        s.ens.configure(E.leja_opts(tol=1e-6))
        s.T = [torch.empty_like(f.T0) for f in s.f]
        return s
    f = s.f = Fields(c, seed)
    if c["op"] == "gradient":
        g = _gen(seed + 7)
        obs = torch.sort(torch.randperm(f.N, generator=g, device=DEV)[:16])[0]
        data = 20.0 + 60.0 * torch.rand((16,), generator=g, device=DEV, dtype=F64)
        s.model = MisfitModel(f.dim, f.nx, f.ny, f.nz, f.phys, f.phi, f.lam, f.dt, c["steps"], obs, data,
                              precision=c["precision"], checkpoint=4)
        s.lnk, s.T0 = f.lnk.clone().requires_grad_(True), f.T0.clone().requires_grad_(True)
        return s
    s.ctx = E.Context(f.dim, f.nx, f.ny, f.nz, physics=f.phys, precision=c["precision"])
    s.T = f.T0.clone()
    if c["op"] == "pressure":
        s.p = torch.empty_like(f.p)
        return s
    if c["op"] == "coupled":  # the pressure of the previous step's temperature
        s.p0 = f.p
        s.ctx.pressure_solve(f.lnk, 0.98 * f.T0 + 0.5, s.p0, tol=1e-10)
        s.p = s.p0.clone()
        return s
    if f.phys.fluid_model or c["field"] == "gauss":
        s.ctx.pressure_solve(f.lnk, f.T0 if f.phys.fluid_model else None, f.p, tol=PTOL)
    if c["op"] == "phi1":
        g = _gen(seed + 9)
        s.v = _gauss(f.shape, 0.05, 1.0, g)
        s.out = torch.empty_like(s.v)
    elif c["op"] not in ("ros2", "ros3p"):
        s.ctx.set_state(f.T0, f.p, f.lnk, f.phi, f.lam, f.dt)
    return s


def run(s):
    c, f = s.case, s.f
    op = c["op"]
    if op == "ensemble":
        for e, fe in enumerate(f):
            s.ens.set_temperature(e, fe.T0)
        s.ens.run(c["steps"])
        for e in range(len(f)):
            s.ens.get_member(e, s.T[e])
        return s.T
    if op == "gradient":
        L = misfit(s.lnk, s.T0, s.model)
        gk, gT = torch.autograd.grad(L, [s.lnk, s.T0])
        return {"L": L, "lnk": gk, "T0": gT}
    if op == "pressure":
        s.p.copy_(f.p)
        s.ctx.pressure_solve(f.lnk, None, s.p)
        return s.p
    if op == "phi1":
        s.ctx.set_state(f.T0, f.p, f.lnk, f.phi, f.lam, f.dt)
        s.ctx.phi1_apply(s.v, s.out)
        return s.out
    s.T.copy_(f.T0)
    if op == "coupled":
        s.p.copy_(s.p0)
        for _ in range(c["steps"]):
            s.ctx.coupled_step(s.T, s.p, f.lnk, f.phi, f.lam, f.dt)
        return {"T": s.T, "p": s.p}
    for _ in range(c["steps"]):
        if op == "steps":
            s.ctx.erem_step(s.T, f.dt)
        elif op == "forced":
            s.ctx.erem_step_forced(s.T, f.dt, *FORCED)
        elif op == "krylov":
            s.ctx.erem_step_krylov(s.T, f.dt)
        else:
            s.ctx.rosm_step(s.T, f.dt, scheme=E.EREM_ROS3P if op == "ros3p" else E.EREM_ROS2,
                            p=f.p, lnk=f.lnk, phi=f.phi, lam=f.lam)
    return s.T


def work(case):
    """Bytes: the inputs of every call read once and its outputs written once
    (a step reads the operator, 7 or 5 coefficients a cell of the context's
    precision, and T, and writes T; assembly and solves read their fields).
    Flops: the stencil products and sums of a typical number of Leja terms,
    Krylov passes or solver iterations."""
    c = case
    if c["op"] == "ensemble":
        cells = sum(n * n for n, _ in _members(c, 0))
    else:
        cells = c["nx"] * c["ny"] * c["nz"]
    nc = 7 if c["nz"] > 1 else 5
    es = 4 if c["precision"] == "fp32_bulk" else 8
    step = cells * (nc * es + 16)
    terms = {"steps": 30, "phi1": 30, "forced": 60, "krylov": 90, "coupled": 250, "ros2": 200, "ros3p": 300,
             "ensemble": 100, "gradient": 90, "pressure": 200}[c["op"]]
    if c["op"] in ("phi1", "coupled", "ros2", "ros3p"):  # fields: p, ln K, phi, lambda
        step += cells * 32
    if c["op"] == "pressure":
        step = cells * 24
    return {"bytes": float(step * c["steps"]), "flops": float(cells * c["steps"] * terms * 2 * nc)}


# ---------------------------------------------------------------------------
# FP64 results in torch
# ---------------------------------------------------------------------------
def _harm(area, h, a, b):
    d = 0.5 * h
    den = a * d + b * d
    return torch.where(den != 0, area * a * b / den, torch.zeros_like(den))


class Grid:
    def __init__(self, f):
        self.f, self.shape = f, f.shape
        self.hx, self.hy = 1.0 / f.nx, 1.0 / f.ny
        self.hz = 1.0 / f.nz if f.dim == 3 else 1.0
        self.area = (self.hy * self.hz, self.hx * self.hz, self.hx * self.hy)
        self.vol = self.hx * self.hy * self.hz

    def faces(self, k):
        """Harmonic transmissibilities of a cell field through the inner faces of x, y, z."""
        k = k.reshape(self.shape)
        out = [_harm(self.area[0], self.hx, k[:, :, :-1], k[:, :, 1:]),
               _harm(self.area[1], self.hy, k[:, :-1], k[:, 1:]), _harm(self.area[2], self.hz, k[:-1], k[1:])]
        return out, 2.0 * self.area[0] * k[:, :, 0] / self.hx, 2.0 * self.area[0] * k[:, :, -1] / self.hx


def _rho(T, fm):
    return 1.0 - 3e-4 * (T - 20.0) if fm else torch.ones_like(T)


def _mu(T, fm):
    return torch.exp(-0.02 * (T - 20.0)) if fm else torch.ones_like(T)


def _sl(axis, a, b):
    s = [slice(None)] * 3
    s[axis] = slice(a, b)
    return tuple(s)


def _pressure(G, lnk, T, fm, hl, hr):
    """Steady pressure by Jacobi CG to the limit of FP64."""
    T = T.reshape(G.shape)
    m = torch.exp(lnk).reshape(G.shape) * _rho(T, fm) / _mu(T, fm)
    U, u0, u1 = G.faces(m)
    D = torch.zeros(G.shape, device=DEV, dtype=F64)
    for ax, a in ((0, U[2]), (1, U[1]), (2, U[0])):
        D[_sl(ax, None, -1)] += a
        D[_sl(ax, 1, None)] += a
    D[:, :, 0] += u0
    D[:, :, -1] += u1
    b = torch.zeros_like(D)
    b[:, :, 0] += u0 * hl
    b[:, :, -1] += u1 * hr

    def A(x):
        y = D * x
        for ax, a in ((0, U[2]), (1, U[1]), (2, U[0])):
            y[_sl(ax, None, -1)] -= a * x[_sl(ax, 1, None)]
            y[_sl(ax, 1, None)] -= a * x[_sl(ax, None, -1)]
        return y

    x = (hl + (hr - hl) * _centres(G.shape[2])).expand(G.shape).clone()
    for _ in range(2):  # a restart removes the drift of the recursive residual
        r = b - A(x)
        z = r / D
        p, rz, bb = z.clone(), (r * z).sum(), (b * b).sum()
        for k in range(20000):
            q = A(p)
            al = rz / (p * q).sum()
            x += al * p
            r -= al * q
            z = r / D
            rn = (r * z).sum()
            p = z + (rn / rz) * p
            rz = rn
            if k % 50 == 49 and float((r * r).sum()) <= 1e-28 * float(bb):
                break
    return x


class Heat:
    """The semi-discrete heat equation at a temperature: J (one array per
    neighbour) and G(T), fluxes from the pressure p and the viscosity of T."""

    def __init__(self, f, p, T):
        G, ph = Grid(f), f.phys
        fm, sh = ph.fluid_model, f.shape
        T, p = T.reshape(sh), p.reshape(sh)
        mob = torch.exp(f.lnk).reshape(sh) / _mu(T, fm)
        L, l0, _ = G.faces(f.lam)
        U, u0, u1 = G.faces(mob)
        X, dX = _rho(T, fm) * T, _rho(T, fm) - (3e-4 * T if fm else 0.0)
        ic = 1.0 / ((f.phi * ph.rhoc_f + (1.0 - f.phi) * ph.rhoc_s) * G.vol).reshape(sh)
        self.D = torch.zeros(sh, device=DEV, dtype=F64)
        self.lo, self.hi = [], []
        g = torch.zeros(sh, device=DEV, dtype=F64)
        for ax, l, u in ((0, L[2], U[2]), (1, L[1], U[1]), (2, L[0], U[0])):
            a, b = _sl(ax, None, -1), _sl(ax, 1, None)
            F = ph.rhoc_f * u * (p[a] - p[b])
            up, dn = F.clamp(min=0.0), (-F).clamp(min=0.0)
            self.D[a] -= l + up * dX[a]
            self.D[b] -= l + dn * dX[b]
            self.hi.append((ax, (l + dn * dX[b]) * ic[a]))   # coupling of cell i to i + 1
            self.lo.append((ax, (l + up * dX[a]) * ic[b]))   # coupling of cell i + 1 to i
            q = l * (T[a] - T[b]) + up * X[a] - dn * X[b]
            g[a] -= q
            g[b] += q
        F0, F1 = ph.rhoc_f * u0 * (ph.head_left - p[:, :, 0]), ph.rhoc_f * u1 * (p[:, :, -1] - ph.head_right)
        Tin = torch.tensor(ph.T_inflow, device=DEV, dtype=F64)
        Xin = _rho(Tin, fm) * Tin
        up, dn = F0.clamp(min=0.0), (-F0).clamp(min=0.0)
        self.D[:, :, 0] -= l0 + dn * dX[:, :, 0]
        self.D[:, :, -1] -= F1 * dX[:, :, -1]
        g[:, :, 0] += l0 * (Tin - T[:, :, 0]) + up * Xin - dn * X[:, :, 0]
        g[:, :, -1] -= F1 * X[:, :, -1]
        self.inflow = (l0 + up) * ic[:, :, 0]   # dG/dT_in at the x = 0 cells (linear model)
        self.D *= ic
        self.G = g * ic
        self.norm = 2.0 * float(self.D.abs().max())

    def apply(self, x, transposed=False):
        y = self.D * x
        for (ax, h), (_, l) in zip(self.hi, self.lo):
            if h.numel() == 0:
                continue
            a, b = _sl(ax, None, -1), _sl(ax, 1, None)
            if transposed:
                h, l = l, h
            y[a] += h * x[b]
            y[b] += l * x[a]
        return y

    def solve_ode(self, g, tau, w=None, y=None, transposed=False):
        """y(tau) of y' = J y + g + t w, y(0) = y or 0, by Taylor steps."""
        n = max(1, math.ceil(self.norm * tau / 4.0))
        h = tau / n
        y = torch.zeros_like(self.D) if y is None else y
        for k in range(n):
            d = self.apply(y, transposed)
            if g is not None:
                d = d + g
            if w is not None:
                d = d + (k * h) * w
            t = h * d
            y = y + t
            for j in range(2, 36):
                t = (h / j) * self.apply(t, transposed)
                if j == 2 and w is not None:
                    t = t + (0.5 * h * h) * w
                y = y + t
        return y


def _stage_solve(H, sigma, b):
    """(sigma I - J) x = b by Jacobi BiCGSTAB."""
    M = 1.0 / (sigma - H.D)

    def A(x):
        return sigma * x - H.apply(x)

    x = M * b
    for _ in range(3):
        r = b - A(x)
        if float(r.norm()) <= 1e-15 * float(b.norm()):
            break
        rh, p, v = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
        rho = al = om = torch.ones((), device=DEV, dtype=F64)
        stop = 1e-14 * float(b.norm())
        for k in range(3000):
            rn = (rh * r).sum()
            p = r + (rn / rho) * (al / om) * (p - om * v)
            y = M * p
            v = A(y)
            al = rn / (rh * v).sum()
            s = r - al * v
            z = M * s
            t = A(z)
            om = (t * s).sum() / (t * t).sum()
            x = x + al * y + om * z
            r = s - om * t
            rho = rn
            if k % 5 == 4 and float(r.norm()) <= stop:
                break
    return x


def _rosm(f, H, p, T, dt, scheme):
    """One ROS2(1) or ROS3p step: (I/(dt g) - J) k_i = G(Y_i) - sum_j c_ij k_j / dt."""
    if scheme == "ros2":
        g = 1.0 + 1.0 / math.sqrt(2.0)
        a, cc, b = [[], [1.0 / g]], [[], [2.0 / g]], [1.5 / g, 0.5 / g]
    else:
        r3 = math.sqrt(3.0)
        g = (3.0 + r3) / 6.0
        a = [[], [1.0 / g], [1.0 / g, 0.0]]
        cc, b = [[], [1.0 / (g * g)], [2.0 * r3, r3]], [2.0, 1.0 / r3, 1.0 - 1.0 / r3]
    T, ks = T.reshape(f.shape), []
    for i in range(len(b)):
        Y = T + sum(w * k for w, k in zip(a[i], ks))
        rhs = _G(f, H, p, T, Y) - sum(w * k for w, k in zip(cc[i], ks)) / dt
        ks.append(_stage_solve(H, 1.0 / (dt * g), rhs))
    return T + sum(w * k for w, k in zip(b, ks))


def _G(f, H, p, T, Y):
    """G at Y with the Darcy fluxes (viscosity) of T."""
    if Y is T:
        return H.G
    fm = f.phys.fluid_model
    mob = f.lnk - torch.log(_mu(T, fm)).reshape(-1) + torch.log(_mu(Y, fm)).reshape(-1)
    keep, f.lnk = f.lnk, mob   # K / mu(T) written as K' / mu(Y)
    try:
        return Heat(f, p, Y).G
    finally:
        f.lnk = keep


def _flat(x):
    return x.reshape(-1)


def exact(case, seed):
    c, op = case, case["op"]
    if op == "ensemble":  # the first small members; the others are the same computation
        out = []
        for e, (n, sd) in enumerate(_members(c, seed)):
            if e >= 4 or n > 200:
                out.append(None)
                continue
            f = Fields(c, sd, n, n)
            p = _pressure(Grid(f), f.lnk, f.T0, 0, 1.0, 0.0)
            H = Heat(f, p, f.T0)
            out.append(_flat(f.T0.reshape(f.shape) + H.solve_ode(H.G, c["steps"] * f.dt)))
        return out
    f = Fields(c, seed)
    ph, tau = f.phys, c["steps"] * f.dt
    if op == "pressure":
        return _flat(_pressure(Grid(f), f.lnk, f.T0, 0, ph.head_left, ph.head_right))
    if c["field"] == "layers":
        p = f.p
    else:
        p = _pressure(Grid(f), f.lnk, f.T0, ph.fluid_model, ph.head_left, ph.head_right)
    H = Heat(f, p, f.T0)
    T0 = f.T0.reshape(f.shape)
    if op == "phi1":
        v = _gauss(f.shape, 0.05, 1.0, _gen(seed + 9)).reshape(f.shape)
        return _flat(H.solve_ode(v, f.dt))
    if op in ("steps", "krylov"):
        return _flat(T0 + H.solve_ode(H.G, tau))
    if op == "coupled":
        return {"T": _flat(T0 + H.solve_ode(H.G, f.dt)), "p": _flat(p)} if c["steps"] == 1 else None
    if op in ("ros2", "ros3p"):
        return _flat(_rosm(f, H, p, f.T0, f.dt, op))
    if op == "forced":
        Tin, rate = FORCED
        T = T0
        for _ in range(c["steps"]):  # each step's own inflow temperature and rate
            g = H.apply(T)
            g[:, :, 0] += H.inflow * Tin
            w = torch.zeros_like(g)
            w[:, :, 0] = H.inflow * rate
            T = T + H.solve_ode(g, f.dt, w=w)
        return _flat(T)
    # gradient: the misfit and its derivative with respect to T0 (the flow of
    # the transposed system); the derivative with respect to ln K has no
    # closed form to compare with here
    g = _gen(seed + 7)
    obs = torch.sort(torch.randperm(f.N, generator=g, device=DEV)[:16])[0]
    data = 20.0 + 60.0 * torch.rand((16,), generator=g, device=DEV, dtype=F64)
    TN = _flat(T0 + H.solve_ode(H.G, tau))
    r = TN[obs] - data
    lam = torch.zeros(f.N, device=DEV, dtype=F64)
    lam[obs] = 2.0 * r
    gT = H.solve_ode(None, tau, y=lam.reshape(f.shape), transposed=True)
    return {"L": (r * r).sum(), "lnk": None, "T0": _flat(gT)}
