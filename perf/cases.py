"""Work that users of this framework have it do, as cases that can be timed and checked.

A case is a dict of plain values.  Its "kind" names the entry point:

* ``step``  -- one time step, ``Simulation.step(1)``, from a given state: what a run does
  over and over.  The state (u, v, w, p, theta_l, q_t on the device) is put into the handle's
  fields, the step runs, and the six fields come back.
* ``solve`` -- one pressure Poisson solve, ``Simulation.poisson_solve``, from a zero guess.
* ``unet_forward``, ``unet_grad`` -- the learned first guess: one inference
  (``UNet.forward``), and one training gradient (``UNet.loss_grad``).

``prepare`` makes the inputs on the device from the seed; ``exact`` gives the outputs in 64 bits
by plain torch: the step from its discretised equations with a direct (Fourier / cosine
transform) Poisson solve, the network by ``conv3d`` and autograd.
"""
import math

import numpy as np
import torch

from paper_2301_04698_gb300 import inputs, les

FIELDS = ("u", "v", "w", "p", "theta_l", "q_t")


def listed():
    return [
        # The paper's density current (Sec. 3) at 200 m, FP64: a 2-D validation run of small, many
        # steps -- the smallest grid a user steps, bound by latency.
        {"name": "bubble_256x4x32_fp64", "kind": "step", "case": "bubble", "nx": 256, "ny": 4, "nz": 32,
         "precision": 64, "tol": 1e-10},
        # The parity box, and the box the learned first guess is trained on: 32^3 Taylor-Green in FP64.
        {"name": "tgv_32x32x32_fp64", "kind": "step", "case": "tgv", "nx": 32, "ny": 32, "nz": 32,
         "precision": 64, "tol": 1e-10},
        # A small moist boundary layer in FP64, every physics term on: development and verification runs.
        {"name": "cbl_64x64x48_fp64", "kind": "step", "case": "cbl", "nx": 64, "ny": 64, "nz": 48,
         "precision": 64, "tol": 1e-10},
        # The moist capped boundary layer of the benchmark's second record, FP32.
        {"name": "cbl_128x128x96_fp32", "kind": "step", "case": "cbl", "nx": 128, "ny": 128, "nz": 96,
         "precision": 32, "tol": 1e-6},
        # The same physics on a grid that no tile divides: the size a user types in.
        {"name": "cbl_100x76x61_fp32", "kind": "step", "case": "cbl", "nx": 100, "ny": 76, "nz": 61,
         "precision": 32, "tol": 1e-6},
        # The largest member of the uneven ensemble: does not fit on chip.
        {"name": "cbl_192x192x128_fp32", "kind": "step", "case": "cbl", "nx": 192, "ny": 192, "nz": 128,
         "precision": 32, "tol": 1e-6},
        # WENO3 and the paper's own solver, weighted Jacobi with a fixed number of sweeps.
        {"name": "weno_jacobi_256x256x64_fp32", "kind": "step", "case": "cbl", "nx": 256, "ny": 256, "nz": 64,
         "precision": 32, "tol": 1e-6, "advection": "weno3", "solver": "jacobi", "maxit": 20},
        # The Taylor-Green tiling of the benchmark's default record, at an eighth of its size.
        {"name": "tgv_768x768x128_fp32", "kind": "step", "case": "tgv", "nx": 768, "ny": 768, "nz": 128,
         "precision": 32, "tol": 1e-6},
        # A single solve of an ensemble's smallest member's size, as a caller of the solver alone does it.
        {"name": "solve_64x64x64_fp32", "kind": "solve", "nx": 64, "ny": 64, "nz": 64, "walls": True,
         "precision": 32, "tol": 1e-6},
        # A single FP64 solve that streams through memory.
        {"name": "solve_256x256x128_fp64", "kind": "solve", "nx": 256, "ny": 256, "nz": 128, "walls": True,
         "precision": 64, "tol": 1e-8},
        # One inference of the learned first guess on its training box: one per Poisson solve.
        {"name": "unet_forward_32_b1", "kind": "unet_forward", "n": 32, "batch": 1},
        # One training gradient at the training batch.
        {"name": "unet_grad_32_b16", "kind": "unet_grad", "n": 32, "batch": 16},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("tgv", "tgv", "cbl", "cbl", "cbl", "bubble", "solve", "solve", "unet_forward", "unet_grad"))
    if kind in ("unet_forward", "unet_grad"):
        n = 4 * _spread(rng, 4, 16)
        batch = rng.randint(1, max(1, min(16, 16 * 32 ** 3 // n ** 3)))
        while 0 < (n // 4) ** 3 * batch % 64 < 16:  # the last, partial tile of the coarsest level
            batch -= 1
        return {"kind": kind, "n": n, "batch": batch}
    precision = rng.choice((32, 32, 64))
    if kind == "bubble":
        nx = _spread(rng, 100, 512)
        return {"kind": "step", "case": "bubble", "nx": nx, "ny": 4, "nz": max(12, nx // 8), "precision": precision,
                "tol": 1e-10 if precision == 64 else 1e-6}
    # whole tiles as often as not
    unit = rng.choice((1, 1, 16, 32, 64))
    most = 256 if precision == 64 else 512
    nx, ny = (max(unit, _spread(rng, 32, most) // unit * unit) for _ in range(2))
    nz = _spread(rng, 24, 128)
    nx, ny = max(nx, 16), max(ny, 16)
    if kind == "solve":
        return {"kind": "solve", "nx": nx, "ny": ny, "nz": nz, "walls": rng.random() < 0.5, "precision": precision,
                "tol": 1e-8 if precision == 64 else 1e-6}
    c = {"kind": "step", "case": kind, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
         "tol": 1e-10 if precision == 64 else 1e-6}
    if rng.random() < 0.3:
        c["advection"] = "weno3"
    if rng.random() < 0.3:
        c.update(solver="jacobi", maxit=rng.randint(5, 40))
    return c


def work(case):
    """Bytes: every input read once and every output written once.  Flops: the arithmetic of one pass that
    does not depend on how often the solver iterates (face values, stresses, fluxes; the convolutions)."""
    if case["kind"].startswith("unet"):
        n3, b = case["n"] ** 3, case["batch"]
        per = sum(2 * ci * co * k ** 3 * n3 // 8 ** lev for ci, co, k, lev in _LAYERS)
        if case["kind"] == "unet_forward":
            return {"bytes": 8 * n3 * b + 4 * _NPARAM, "flops": per * b}
        return {"bytes": 8 * n3 * b + 8 * _NPARAM, "flops": 3 * per * b}
    cells, es = case["nx"] * case["ny"] * case["nz"], case["precision"] // 8
    if case["kind"] == "solve":
        return {"bytes": 2 * cells * es, "flops": 30 * cells}
    sweeps = case.get("maxit", 0) if case.get("solver") == "jacobi" else 0
    return {"bytes": 12 * cells * es, "flops": 3 * (700 + 12 * sweeps) * cells}


# ---- inputs ----------------------------------------------------------------------------------------


def _case(c):
    """The workload as the framework describes it (paper_2301_04698_gb300.inputs)."""
    kw = dict(precision=c["precision"], tol=c["tol"], maxit=c.get("maxit", 20000),
              advection=c.get("advection", "quick"), solver=c.get("solver", "cg"))
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if c["kind"] == "solve":
        return inputs.Case("solve", nx, ny, nz, 35.0, 35.0, 960.0 / nz, walls=c["walls"], rho0_const=1.0, **kw)
    if c["case"] == "tgv":  # 32 nodes a period
        tol = kw.pop("tol")
        return inputs.tgv(32, nxyz=(nx, ny, nz), steps_tol=tol, dt=0.3 / 64, **kw)
    if c["case"] == "cbl":  # the domain's height as in the 96-level boundary layer
        return inputs.cbl(nx, ny, nz, dz=960.0 / nz, **kw)
    base = inputs.density_current(51200.0 / nx, ny=ny, precision=c["precision"])
    return base.replace(nx=nx, ny=ny, nz=nz, **kw)


def _waves(case, gen, amp, count=5, vary_y=True):
    """A smooth random field: a few long waves."""
    dev = gen.device
    r = torch.rand(count, 6, generator=gen, device=dev, dtype=torch.float64).cpu().numpy()
    f = torch.zeros(case.shape, device=dev, dtype=torch.float64)
    x = torch.arange(case.nx, device=dev, dtype=torch.float64) / case.nx
    y = torch.arange(case.ny, device=dev, dtype=torch.float64) / case.ny
    z = (torch.arange(case.nz, device=dev, dtype=torch.float64) + 0.5) / case.nz
    for q in range(count):
        a, kx, ky = amp * (r[q, 0] + 0.5) / count, 1 + int(4 * r[q, 1]), int(4 * r[q, 2]) if vary_y else 0
        kz = 1 + int(3 * r[q, 3])
        hx = torch.exp(2j * math.pi * (kx * x + r[q, 4]))
        hy = torch.exp(2j * math.pi * (ky * y)) * a
        plane = (hy[:, None] * hx[None, :]).real
        if case.walls:
            col = torch.cos(math.pi * kz * z)
        else:
            col = torch.cos(2 * math.pi * (kz * z + r[q, 5]))
        f += col[:, None, None] * plane[None]
    return f


def _noise(case, gen, amp):
    return (2.0 * torch.rand(case.shape, generator=gen, device=gen.device, dtype=torch.float64) - 1.0) * amp


def _state(c, seed):
    """u, v, w, p, theta_l, q_t in the case's precision, on the device."""
    case = _case(c)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    dev, f64 = gen.device, torch.float64
    z = (torch.arange(case.nz, device=dev, dtype=f64) + 0.5) * case.dz
    one = torch.ones(case.shape, device=dev, dtype=f64)
    s = {}
    if c["case"] == "tgv":
        x = 2 * math.pi * (torch.arange(case.nx, device=dev, dtype=f64) + 0.5) * case.dx
        y = 2 * math.pi * (torch.arange(case.ny, device=dev, dtype=f64) + 0.5) * case.dy
        zz = torch.cos(2 * math.pi * z)[:, None, None]
        s["u"] = zz * (torch.sin(x)[None, :] * torch.cos(y)[:, None]) + _noise(case, gen, 0.02)
        s["v"] = -zz * (torch.cos(x)[None, :] * torch.sin(y)[:, None]) + _noise(case, gen, 0.02)
        s["w"] = _noise(case, gen, 0.02)
        s["p"] = _waves(case, gen, 0.05)
        s["theta_l"] = 300.0 * one + _waves(case, gen, 0.5)
        s["q_t"] = 0.002 * one + _waves(case, gen, 0.001)
    elif c["case"] == "cbl":  # a layer that turns: waves and noise below a seeded inversion
        zi = 960.0 * (0.7 + 0.2 * float(torch.rand(1, generator=gen, device=dev)))
        below = (z < zi).to(f64)[:, None, None]
        s["u"] = case.ug + _waves(case, gen, 0.6) + _noise(case, gen, 0.1) * below
        s["v"] = case.vg + _waves(case, gen, 0.6) + _noise(case, gen, 0.1) * below
        s["w"] = (_waves(case, gen, 0.6) + _noise(case, gen, 0.1)) * below
        s["p"] = _waves(case, gen, 1.0)
        s["theta_l"] = 289.0 + 7.5 * (1 - below) + (_waves(case, gen, 0.3) + _noise(case, gen, 0.1)) * below
        s["q_t"] = 9e-3 - 6.5e-3 * (1 - below) + _waves(case, gen, 4e-4) * below
    else:  # a cold bubble of a seeded place and strength, in slow motion; the same on every y
        a, r = case.init_args, torch.rand(3, generator=gen, device=dev, dtype=f64).cpu().numpy()
        x = (torch.arange(case.nx, device=dev, dtype=f64) + 0.5) * case.dx
        d = torch.sqrt(((x[None, :] - a["xc"] - 4000 * (r[0] - 0.5)) / a["xr"]) ** 2 +
                       ((z[:, None] - a["zc"]) / a["zr"]) ** 2).clamp(max=1.0)
        th = (-10.0 - 10.0 * r[1]) * torch.cos(0.5 * math.pi * d) ** 2
        s["theta_l"] = 300.0 + th[:, None, :] * one
        s["u"] = _waves(case, gen, 4.0, vary_y=False)
        s["w"] = _waves(case, gen, 4.0, vary_y=False)
        s["v"] = 0.0 * one
        s["p"] = _waves(case, gen, 20.0, vary_y=False)
        s["q_t"] = 0.0 * one
    dt = torch.float64 if case.precision == 64 else torch.float32
    return {k: s[k].to(dt).contiguous() for k in FIELDS}


def _rhs(c, seed):
    """A right side as a step forms it: the central divergence of a velocity of waves and noise."""
    case = _case(c)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    b = torch.zeros(case.shape, device=gen.device, dtype=torch.float64)
    for d in range(3):
        f = _waves(case, gen, 1.0) + _noise(case, gen, 0.1)
        h = (case.dx, case.dy, case.dz)[d]
        b += (_sh(case, f, d, 1, 1) - _sh(case, f, d, -1, 1)) / (2 * h)
    return b.to(torch.float64 if case.precision == 64 else torch.float32)


_LAYERS = ((1, 16, 3, 0), (16, 16, 3, 0), (16, 32, 3, 1), (32, 32, 3, 1), (32, 64, 3, 2), (64, 64, 3, 2),
           (96, 32, 3, 1), (32, 32, 3, 1), (48, 16, 3, 0), (16, 16, 3, 0), (16, 1, 1, 0))  # cin, cout, k, level
_NPARAM = sum(ci * co * k ** 3 + co for ci, co, k, _ in _LAYERS)


def _unet_data(c, seed):
    """Weights as after initialisation, right sides b and solutions psi (b's long waves)."""
    rng = np.random.default_rng(int(seed))
    w = []
    for ci, co, k, _ in _LAYERS:
        w += [rng.standard_normal(ci * co * k ** 3) * math.sqrt(2.0 / (ci * k ** 3)), 0.05 * rng.standard_normal(co)]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n, batch = c["n"], c["batch"]
    box = inputs.tgv(32, nxyz=(n, n, n))
    psi = torch.stack([_waves(box, gen, 1.0) for _ in range(batch)])
    b = 20.0 * psi + torch.rand(psi.shape, generator=gen, device="cuda", dtype=torch.float64) - 0.5
    return np.concatenate(w).astype(np.float32), b.float(), (1e-3 * psi).float()


# ---- the cases -------------------------------------------------------------------------------------


def prepare(case, seed):
    if case["kind"].startswith("unet"):
        w, b, psi = _unet_data(case, seed)
        net = les.UNet(case["n"], max_batch=case["batch"])
        net.set_weights(w)
        net.out_scale = 1e-3
        return {"kind": case["kind"], "net": net, "b": b, "psi": psi}
    sim = les.Simulation(_case(case))
    if case["kind"] == "solve":
        return {"kind": "solve", "sim": sim, "b": _rhs(case, seed), "tol": case["tol"]}
    return {"kind": "step", "sim": sim, "state": _state(case, seed)}


def run(state):
    kind = state["kind"]
    if kind == "unet_forward":
        return {"psi0": state["net"].forward(state["b"])}
    if kind == "unet_grad":
        loss, grad = state["net"].loss_grad(state["b"], state["psi"])
        return {"loss": loss, "grad": grad}
    sim = state["sim"]
    if kind == "solve":
        x = torch.zeros_like(state["b"])
        sim.poisson_solve(state["b"], x, state["tol"], 20000)
        return {"x": x}
    for k in FIELDS:
        sim.view(k).copy_(state["state"][k])
    sim.step(1, allow_not_converged=True)  # a fixed number of Jacobi sweeps ends without converging
    return {k: sim.view(k) for k in FIELDS}


# ---- the same in 64 bits ---------------------------------------------------------------------------

_RD, _RV, _CPD, _CPV, _CL, _LV, _G = 287.0, 461.89, 1004.5, 1859.5, 4181.0, 2.47e6, 9.81


def _sh(case, f, d, n, ghost):
    """f at the node n steps further along d.  Ghosts beyond walls: 0 even, 1 odd, 2 horizontal velocity
    (even at the surface, odd at the lid)."""
    if d < 2:
        return torch.roll(f, -n, 2 - d)
    if not case.walls:
        return torch.roll(f, -n, 0)
    k = torch.arange(case.nz, device=f.device) + n
    lo, hi = k < 0, k >= case.nz
    k = torch.where(lo, -1 - k, torch.where(hi, 2 * case.nz - 1 - k, k))
    s = torch.ones(case.nz, device=f.device, dtype=f.dtype)
    if ghost == 1:
        s[lo] = -1.0
    if ghost:
        s[hi] = -1.0
    return f[k] * s[:, None, None] if f.dim() == 3 else f[k] * s


def _weno(a, b, c):
    m = torch.maximum(a.abs(), torch.maximum(b.abs(), c.abs()))
    eps = 1e-6 * m * m + 1e-18
    a0, a1 = 1 / (3 * (eps + (b - a) ** 2) ** 2), 2 / (3 * (eps + (c - b) ** 2) ** 2)
    return (a0 * 0.5 * (3 * b - a) + a1 * 0.5 * (b + c)) / (a0 + a1)


class _Exact:
    """One step of a case from its discretised equations, every field in 64 bits."""

    def __init__(self, case, dev):
        self.c, self.dev = case, dev
        z = (torch.arange(case.nz, device=dev, dtype=torch.float64) + 0.5) * case.dz
        self.z = z[:, None, None]
        p0 = case.p00 * (1 - _G * z / (_CPD * case.theta0)) ** (_CPD / _RD)
        rho = p0 / (_RD * case.theta0 * (p0 / case.p00) ** (_RD / _CPD))
        if case.rho0_const is not None:
            rho = torch.full_like(z, case.rho0_const)
        self.p0, self.rho = p0[:, None, None], rho[:, None, None]
        self.h = (case.dx, case.dy, case.dz)

    def on(self, name):
        return name in self.c.physics

    def sh(self, f, d, n, ghost=0):
        return _sh(self.c, f, d, n, ghost)

    def face(self, f, F, d, ghost):
        a, c, e = self.sh(f, d, -1, ghost), self.sh(f, d, 1, ghost), self.sh(f, d, 2, ghost)
        if self.c.advection == "weno3":
            return torch.where(F >= 0, _weno(a, f, c), _weno(e, c, f))
        return torch.where(F >= 0, (6 * f - a + 3 * c) / 8, (3 * f + 6 * c - e) / 8)

    def flux(self, ud, d, ghost):
        """Mass flux through the upper face of each node along d."""
        r = self.rho * ud
        return 0.5 * (r + self.sh(r, d, 1, ghost))

    def div(self, up, d, bottom):
        """Difference over a node of its faces' fluxes; bottom: through the surface."""
        low = torch.roll(up, 1, 2 - d)
        if d == 2 and self.c.walls:
            low[0] = bottom
        return (up - low) / self.h[d]

    def nu(self, vel, b):
        c = self.c
        if self.on("const_nu") or not self.on("sgs"):
            return torch.full_like(vel[0], c.nu_const if self.on("const_nu") else 0.0)
        gh = (2, 2, 1)
        g = [[(self.sh(vel[q], d, 1, gh[q]) - self.sh(vel[q], d, -1, gh[q])) / (2 * self.h[d]) for d in range(3)]
             for q in range(3)]
        s2 = 0
        for q in range(3):
            for d in range(3):
                s2 = s2 + 0.5 * (g[q][d] + g[d][q]) ** 2
        out = (c.cs * (c.dx * c.dy * c.dz) ** (1 / 3)) ** 2 * torch.sqrt(s2)
        if self.on("fb"):
            n2 = (self.sh(b, 2, 1) - self.sh(b, 2, -1)) / (2 * c.dz)
            out = out * torch.sqrt((1 - n2 / (c.pr * s2)).clamp(0, 1))
        return out

    # moist thermodynamics
    def rm(self, qt, ql):
        return (1 - qt) * _RD + (qt - ql) * _RV

    def cpm(self, qt, ql):
        return (1 - qt) * _CPD + (qt - ql) * _CPV + ql * _CL

    def exner(self, qt, ql):
        return (self.p0 / self.c.p00) ** (self.rm(qt, ql) / self.cpm(qt, ql))

    def qsat(self, t):
        es = 611.657 * torch.exp(_LV / _RV * (1 / 273.16 - 1 / t))
        e = _RD / _RV
        return e * es / (self.p0 - (1 - e) * es)

    def thermo(self, th, qt):
        c = self.c
        t = self.exner(qt, 0 * qt) * th
        ql = torch.zeros_like(t)
        if self.on("moist"):
            def f(x):
                q = (qt - self.qsat(x)).clamp(min=0)
                return x / self.exner(qt, q) * (1 - _LV * q / (self.cpm(qt, q) * x)) - th
            wet = qt > self.qsat(t)
            ta, tb = t, t + _LV * (qt - self.qsat(t)) / self.cpm(qt, 0 * qt)
            fa, fb = f(ta), f(tb)
            for _ in range(12):
                go = (fb.abs() > 1e-12) & (fb != fa)
                tc = torch.where(go, tb - fb * (tb - ta) / torch.where(fb == fa, torch.ones_like(fb), fb - fa), tb)
                ta, fa, tb = tb, fb, tc
                fb = f(tb)
            t = torch.where(wet, tb, t)
            ql = torch.where(wet, (qt - self.qsat(t)).clamp(min=0), ql)
        b = _G * (self.rm(qt, ql) * t / self.p0 * self.rho - 1) if self.on("buoy") else torch.zeros_like(t)
        rad = torch.zeros_like(t)
        if self.on("rad"):
            below = torch.cumsum(self.rho * ql * c.dz, 0)
            total = below[-1:]
            up = c.rad_f0 * torch.exp(-c.rad_kappa * (total - below)) + c.rad_f1 * torch.exp(-c.rad_kappa * below)
            low = torch.cat((c.rad_f0 * torch.exp(-c.rad_kappa * total) + c.rad_f1, up[:-1]))
            rad = -(up - low) / c.dz / (self.cpm(qt, ql) * self.exner(qt, ql))
        return b, rad

    def scalar(self, vel, phik, phih, pr, bottom, nu, rad):
        c, f = self.c, 0.5 * (phik + phih)
        tend = rad
        for d in range(3):
            r = 0.5 * (self.rho + self.sh(self.rho, 2, 1)) if d == 2 else self.rho
            up = r * 0.5 * (nu + self.sh(nu, d, 1)) / pr * (self.sh(f, d, 1) - f) / self.h[d]
            if self.on("adv"):
                F = self.flux(vel[d], d, (2, 2, 1)[d])
                up = up - F * self.face(f, F, d, 0)
            if d == 2 and c.walls:
                up[-1] = 0.0
            tend = tend + self.div(up, d, bottom)
        if self.on("subs"):
            tend = tend + self.rho * c.subs_div * self.z * (self.sh(f, 2, 1) - f) / c.dz
        return phih + c.dt * tend / self.rho

    def momentum(self, uk, un, p, b):
        c, gh = self.c, (2, 2, 1)
        v = [0.5 * (x + y) for x, y in zip(uk, un)]
        nu = self.nu(v, b)
        ap = p / self.rho
        out = []
        for q in range(3):
            r = 0
            for d in range(3):
                rf = 0.5 * (self.rho + self.sh(self.rho, 2, 1)) if d == 2 else self.rho
                dn = (self.sh(v[q], d, 1, gh[q]) - v[q]) / self.h[d]
                if q == d:
                    dt = dn
                else:  # along q of the component d, at both nodes of the face
                    def along(n):
                        x = self.sh(v[d], d, n, gh[d]) if n else v[d]
                        if q < 2 or not c.walls or d == 2:
                            return (self.sh(x, q, 1, gh[d]) - self.sh(x, q, -1, gh[d])) / (2 * self.h[q])
                        return (self.sh(x, 2, 1, gh[d]) - self.sh(x, 2, -1, gh[d])) / (2 * self.h[q])
                    dt = 0.5 * (along(0) + along(1))
                up = rf * 0.5 * (nu + self.sh(nu, d, 1)) * (dn + dt)
                if self.on("adv"):
                    F = self.flux(v[d], d, gh[d])
                    adv = F * self.face(v[q], F, d, gh[q])
                    if d == 2 and c.walls:
                        adv[-1] = 0.0
                    up = up - adv
                r = r + self.div(up, d, 0.0)
            if self.on("buoy") and q == 2:
                r = r + self.rho * b
            if self.on("coriolis") and q < 2:
                r = r + (c.f_cor * self.rho * (v[1] - c.vg) if q == 0 else -c.f_cor * self.rho * (v[0] - c.ug))
            if self.on("sponge"):
                top = c.nz * c.dz
                zs = (1 - c.sponge_frac) * top
                s = torch.sin(0.5 * math.pi * ((self.z - zs) / (top - zs)).clamp(min=0)) ** 2
                r = r - c.sponge_rate * s * self.rho * (v[q] - (c.ug, c.vg, 0.0)[q])
            gp = (self.sh(ap, q, 1) - self.sh(ap, q, -1)) / (2 * self.h[q])
            out.append(un[q] + c.dt * (r / self.rho - gp))
        return out

    def rhs(self, hat, psi):
        out = 0
        for d in range(3):
            m = self.rho * hat[d]
            g = (2, 2, 1)[d]
            out = out + (self.sh(m, d, 1, g) - self.sh(m, d, -1, g)) / (2 * self.h[d]) / (self.rho * self.c.dt)
            out = out - (self.sh(psi, d, 2) - 4 * self.sh(psi, d, 1) + 6 * psi - 4 * self.sh(psi, d, -1) +
                         self.sh(psi, d, -2)) / (4 * self.h[d] ** 2)
        return out

    def lap(self, x):
        return sum((self.sh(x, d, 1) - 2 * x + self.sh(x, d, -1)) / self.h[d] ** 2 for d in range(3))

    def solve(self, b):
        c, dev = self.c, self.dev
        b = b - b.mean()
        if c.solver == "jacobi":
            dz = torch.full((c.nz, 1, 1), -2.0 / c.dz ** 2, device=dev, dtype=torch.float64)
            if c.walls:
                dz[0], dz[-1] = dz[0] / 2, dz[-1] / 2
            diag = dz - 2 / c.dx ** 2 - 2 / c.dy ** 2
            x = torch.zeros_like(b)
            for _ in range(c.maxit):
                x = x + c.omega * (b - self.lap(x)) / diag
            return x - x.mean()

        def eig(n, h, half):
            k = torch.arange(n, device=dev, dtype=torch.float64)
            return (2 * torch.cos((1 if half else 2) * math.pi * k / n) - 2) / h ** 2
        f = torch.fft.rfft2(b)
        lam = eig(c.ny, c.dy, False)[None, :, None] + eig(c.nx, c.dx, False)[None, None, : f.shape[2]]
        if c.walls:  # cosine modes along z
            k = torch.arange(c.nz, device=dev, dtype=torch.float64)
            m = torch.cos(math.pi * k[:, None] * (k[None, :] + 0.5) / c.nz) * math.sqrt(2 / c.nz)
            m[0] /= math.sqrt(2)
            def along(t, g):
                return torch.complex(torch.tensordot(t, g.real.contiguous(), 1), torch.tensordot(t, g.imag.contiguous(), 1))
            f = along(m, f)
        else:
            f = torch.fft.fft(f, dim=0)
        lam = lam + eig(c.nz, c.dz, c.walls)[:, None, None]
        lam[0, 0, 0] = 1.0
        f /= lam
        f[0, 0, 0] = 0.0
        f = along(m.T, f) if c.walls else torch.fft.ifft(f, dim=0)
        return torch.fft.irfft2(f, s=(c.ny, c.nx))

    def step(self, s):
        c = self.c
        u, p, th, qt = [s["u"], s["v"], s["w"]], s["p"], s["theta_l"], s["q_t"]
        un, thh, qth = list(u), th, qt
        b, rad = self.thermo(th, qt)
        psi = torch.zeros_like(p)
        sfc = self.on("sfc")
        for _ in range(c.K):
            nu = self.nu(u, b)
            th = self.scalar(u, th, thh, c.pr, -c.shf / _CPD if sfc else 0.0, nu, rad)
            qt = self.scalar(u, qt, qth, c.sc, -c.lhf / _LV if sfc else 0.0, nu, 0.0)
            hat = self.momentum(u, un, p, b)
            psi = self.solve(self.rhs(hat, psi))
            u = [hat[d] - c.dt * (self.sh(psi, d, 1) - self.sh(psi, d, -1)) / (2 * self.h[d]) for d in range(3)]
            p = p + self.rho * psi
        return {"u": u[0], "v": u[1], "w": u[2], "p": p, "theta_l": th, "q_t": qt}


def _net(flat, b):
    """The network's output for b (batch, n, n, n) and the scale of each right side."""
    w, o = [], 0
    for ci, co, k, _ in _LAYERS:
        m = ci * co * k ** 3
        w.append((flat[o:o + m].reshape(co, ci, k, k, k), flat[o + m:o + m + co]))
        o += m + co
    nn = torch.nn.functional

    def conv(x, q):
        k = w[q][0].shape[2]
        if k > 1:
            x = nn.pad(x, (1, 1, 1, 1, 1, 1), mode="circular")
        return nn.conv3d(x, *w[q])

    def block(x, q):
        return nn.leaky_relu(conv(nn.leaky_relu(conv(x, q), 0.1), q + 1), 0.1)

    def up(x):
        return x.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)
    s = b.square().mean((1, 2, 3), keepdim=True).sqrt()
    e1 = block((b / s)[:, None], 0)
    e2 = block(nn.avg_pool3d(e1, 2), 2)
    e3 = block(nn.avg_pool3d(e2, 2), 4)
    g2 = block(torch.cat((up(e3), e2), 1), 6)
    g1 = block(torch.cat((up(g2), e1), 1), 8)
    return conv(g1, 10)[:, 0], s


def exact(case, seed):
    if case["kind"].startswith("unet"):
        flat, b, psi = _unet_data(case, seed)
        flat, b, psi = torch.from_numpy(flat).double().cuda(), b.double(), psi.double()
        with torch.backends.cudnn.flags(enabled=False), torch.enable_grad():
            if case["kind"] == "unet_forward":
                y, s = _net(flat, b)
                return {"psi0": s * 1e-3 * (y - y.mean((1, 2, 3), keepdim=True))}
            flat.requires_grad_(True)
            total, grad = 0.0, torch.zeros_like(flat)
            for q in range(b.shape[0]):  # a sample at a time: the unfolded 64-bit convolutions are large
                y, s = _net(flat, b[q:q + 1])
                loss = (y - psi[q:q + 1] / (s * 1e-3)).square().mean() / b.shape[0]
                grad += torch.autograd.grad(loss, flat)[0]
                total += float(loss)
            return {"loss": total, "grad": grad}
    if case["kind"] == "solve":
        return {"x": _Exact(_case(case), "cuda").solve(_rhs(case, seed).double())}
    return _Exact(_case(case), "cuda").step({k: v.double() for k, v in _state(case, seed).items()})
