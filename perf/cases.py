"""Performance cases: the work that users of this framework have it do, each
through the public calls of ``paper_1503_07416_gb300.fm``.

A case is one solver (or one batch of solvers) and one pass of a program that
uses it: the fields of a state are handed over in device memory, a few implicit
time steps are taken (with the energy after each where the program logs it)
and the new fields are read back.  ``exact`` solves the same steps in float64
torch by fixed-point iteration on the scheme's equations, without the library.

Fields of a case:

* ``model``: ``hydro`` (the compressible step), ``gradflow`` (the conservative
  gradient flow) or ``batch`` (many 2-D hydrodynamic instances at once);
* ``kind``: ``pfc`` or ``cdft``; ``dim``, ``nx``, ``ny``, ``nz``: the grid
  (``sizes``: the square sizes of a batch, comma separated); ``h``: spacing;
* ``dt``, ``steps``: step size and steps per pass (``dt_lo``/``dt_hi``: the
  log-uniform range of a batch's step sizes);
* ``prec``: ``mixed`` or ``fp64``; ``w``, ``tol``, ``coarsest``, ``ncoarse``,
  ``extrapolate``: solver options;
* ``walls``: no-slip walls in y moving at -walls / +walls (absent: periodic);
* ``energy``: the energy terms are read after every step.
"""
from __future__ import annotations

import math

import torch

from paper_1503_07416_gb300 import fm, inputs

H_HEX = inputs.H_HEX
PREC = {"mixed": fm.FM_MIXED, "fp64": fm.FM_FP64}
GAMMA = 2.0


def _hydro(name, kind, nx, ny, nz=1, dim=2, **kw):
    c = dict(name=name, model="hydro", kind=kind, dim=dim, nx=nx, ny=ny, nz=nz, h=H_HEX, dt=0.02, steps=4,
             prec="mixed", w=0.0, tol=1e-10, coarsest=16, ncoarse=4, extrapolate=False, energy=False)
    c.update(kw)
    if kind == "pfc":
        c.setdefault("alpha", 0.6)
    return c


def listed():
    return [
        # convergence study, a coarse rung of the refinement path in float64: the smallest calls
        _hydro("conv_pfc32_fp64", "pfc", 32, 32, h=1.0, dt=0.025, prec="fp64", alpha=0.975, tol=1e-12),
        # the same study, CDFT, a middle rung
        _hydro("conv_cdft64_fp64", "cdft", 64, 64, h=0.5, dt=0.00625, prec="fp64", nu=1.0, delta=1e-10, tol=1e-12),
        # freezing run with the library's default cycle and damping, the energy logged every step
        _hydro("freeze_pfc128", "pfc", 128, 128, h=0.25, dt=0.01, alpha=0.975, w=0.5, energy=True),
        # solidification of a 2-D film, the benchmark's hierarchy and initial iterate
        _hydro("film_pfc512", "pfc", 512, 512, steps=8, extrapolate=True, **inputs.BENCH_MG_2D),
        # the same film solved in float64 throughout
        _hydro("film_pfc512_fp64", "pfc", 512, 512, prec="fp64", **inputs.BENCH_MG_2D),
        # a box whose sides are no powers of two (three levels, ragged tiles), default cycle
        _hydro("box_pfc360x200", "pfc", 360, 200),
        # non-local (CDFT) freezing
        _hydro("freeze_cdft256", "cdft", 256, 256, h=34.0 / 256, nu=2.362, delta=1e-10, **inputs.BENCH_MG_2D),
        # a nucleus growing in a 3-D box
        _hydro("nucleus_pfc3d128", "pfc", 128, 128, 128, dim=3, steps=2),
        # a small 3-D box with uneven sides in float64
        _hydro("box_pfc3d40x48x56_fp64", "pfc", 40, 48, 56, dim=3, steps=2, prec="fp64"),
        # an ensemble of films of uneven size and step
        dict(name="ensemble24", model="batch", kind="pfc", dim=2, h=H_HEX, alpha=0.6, dt_lo=1e-3, dt_hi=1e-1, steps=2,
             prec="mixed", w=0.0, tol=1e-10, **inputs.BENCH_MG_2D,
             sizes="1024,128,512,256,128,1024,512,128,256,1024,256,512,128,1024,256,512,512,256,1024,128,256,512,"
                   "1024,128"),
        # conservative gradient flow of the film
        dict(name="flow_pfc512", model="gradflow", kind="pfc", dim=2, nx=512, ny=512, nz=1, h=H_HEX, alpha=0.6, dt=0.02,
             steps=4, prec="mixed", w=0.3, tol=1e-10, **inputs.BENCH_MG_2D),
        # nanocrystal between moving walls, default cycle (the shear study)
        _hydro("shear_pfc256", "pfc", 256, 256, walls=0.1),
    ]


def _even(rng, lo, hi, multiple=2):
    """An even size, log-uniform in [lo, hi]."""
    return max(lo, min(hi, multiple * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple))))


def draw(rng):
    what = rng.choice(("pfc2", "pfc2", "cdft2", "pfc3", "batch", "flow", "walls"))
    prec = rng.choice(("mixed", "mixed", "fp64"))
    mg = rng.choice((dict(coarsest=16, ncoarse=4), dict(coarsest=16, ncoarse=4), dict(coarsest=64, ncoarse=2)))
    dt = round(math.exp(rng.uniform(math.log(2e-3), math.log(5e-2))), 5)
    if what == "pfc2":
        c = _hydro("", "pfc", _even(rng, 32, 640), _even(rng, 32, 640), dt=dt, prec=prec, w=rng.choice((0.0, 0.5)),
                   extrapolate=rng.random() < 0.3, energy=rng.random() < 0.3, **mg)
    elif what == "cdft2":
        n = 2 ** rng.randint(5, 9)
        m = n if rng.random() < 0.5 else 2 ** rng.randint(5, 9)
        h = rng.choice((34.0 / 256, 0.25, 0.5))
        c = _hydro("", "cdft", n, m, h=h, nu=rng.choice((1.0, 2.362)), delta=1e-10, prec=prec,
                   dt=round(dt * min(1.0, h / 0.25), 6), **mg)
    elif what == "pfc3":
        c = _hydro("", "pfc", _even(rng, 16, 112), _even(rng, 16, 112), _even(rng, 16, 112), dim=3, steps=2, dt=dt,
                   prec=prec if prec == "mixed" or rng.random() < 0.5 else "mixed")
        if c["prec"] == "fp64":
            c.update(nx=min(c["nx"], 64), ny=min(c["ny"], 64), nz=min(c["nz"], 64))
    elif what == "batch":
        sizes = [rng.choice((64, 128, 192, 256, 384, 512)) for _ in range(rng.randint(3, 24))]
        c = dict(name="", model="batch", kind="pfc", dim=2, h=H_HEX, alpha=0.6, dt_lo=1e-3, dt_hi=1e-1, steps=2, prec=prec,
                 w=0.0, tol=1e-10, coarsest=64, ncoarse=2, sizes=",".join(map(str, sizes)))
    elif what == "flow":
        c = dict(name="", model="gradflow", kind="pfc", dim=2, nx=_even(rng, 64, 512), ny=_even(rng, 64, 512), nz=1,
                 h=H_HEX, alpha=0.6, dt=min(dt, 0.02), steps=4, prec=prec, w=rng.choice((0.3, 0.5)), tol=1e-10, **mg)
    else:
        c = _hydro("", "pfc", _even(rng, 32, 512), _even(rng, 32, 512), dt=dt, prec=prec, walls=rng.choice((0.0, 0.1)), **mg)
    del c["name"]
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _axis(n, d, dim, dev):
    shape = [1] * dim
    shape[dim - 1 - d] = n
    return torch.arange(n, dtype=torch.float64, device=dev).reshape(shape)


def _fields(kind, ns, h, gen, dev, moving=True, alpha=0.6):
    """A state part of the way through a run, with a smooth slow flow.  PFC
    films (alpha = 0.6): supercooled liquid with noise and Gaussian nuclei; PFC
    at alpha = 0.975 (the freezing and convergence runs, fine grids): smooth
    waves on the solid-forming density; CDFT: the noisy liquid."""
    dim = len(ns)
    shape = tuple(reversed(ns))
    noise = torch.rand(shape, generator=gen, dtype=torch.float64, device=dev)
    par = torch.rand(64, generator=gen, dtype=torch.float64, device=dev).tolist()
    if kind == "cdft":
        rho = 0.1 * math.pi * (1.0 + 0.1 * noise)
    elif alpha > 0.9:
        rho = 1.5 - 0.07 * math.sqrt(3.0) + 1e-4 * (2.0 * noise - 1.0)
        for b in range(6):
            arg = 2.0 * math.pi * par[58 + b]
            for d in range(dim):
                arg = arg + 2.0 * math.pi * (1 + int(4 * par[2 * b + d])) * _axis(ns[d], d, dim, dev) / ns[d]
            rho = rho + 0.02 * torch.sin(arg)
    else:
        rho = 0.80 + 0.01 * (2.0 * noise - 1.0)
        width = inputs.A_ATOM / 2.0
        for b in range(4 if dim == 2 else 1):
            r2 = 0.0
            for d in range(dim):
                x = (_axis(ns[d], d, dim, dev) * h - par[3 * b + d] * ns[d] * h).abs()
                r2 = r2 + torch.minimum(x, ns[d] * h - x) ** 2
            rho = rho + 0.5 * torch.exp(-r2 / (2.0 * width * width))
    vel = []
    for a in range(dim):
        v = torch.zeros(shape, dtype=torch.float64, device=dev)
        for b in range(3 if moving else 0):
            m = 1.0 + int(3 * par[20 + 6 * a + b])
            arg = 0.0
            for d in range(dim):
                arg = arg + (m if (d + b + a) % 2 else 1.0) * 2.0 * math.pi * _axis(ns[d], d, dim, dev) / ns[d]
            v = v + 0.004 * torch.sin(arg + 2.0 * math.pi * par[40 + 6 * a + b])
        vel.append(v.expand(shape).contiguous())
    return rho.contiguous(), vel


def _ns(case):
    return [case["nx"], case["ny"], case["nz"]][: case["dim"]]


def _inputs(case, seed):
    """[(rho, vel, dt)] of the case's instances."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    gen = torch.Generator(device=dev).manual_seed(int(seed) % (1 << 31))
    if case["model"] == "batch":
        out = []
        for n in map(int, case["sizes"].split(",")):
            t = float(torch.rand(1, generator=gen, dtype=torch.float64, device=dev))
            rho, vel = _fields(case["kind"], [n, n], case["h"], gen, dev)
            out.append((rho, vel, math.exp(math.log(case["dt_lo"]) + t * math.log(case["dt_hi"] / case["dt_lo"]))))
        return out
    rho, vel = _fields(case["kind"], _ns(case), case["h"], gen, dev, moving=case["model"] == "hydro",
                       alpha=case.get("alpha", 0.6))
    return [(rho, vel, case["dt"])]


def prepare(case, seed):
    data = _inputs(case, seed)
    stream = torch.cuda.current_stream().cuda_stream
    opts = dict(precision=PREC[case["prec"]], w_damp=case["w"], tol=case["tol"], coarsest=case["coarsest"],
                ncoarse=case["ncoarse"], max_cycles=200, gamma=GAMMA, stream=stream)
    state = dict(case=case, data=data)
    if case["model"] == "batch":
        sizes = [int(n) for n in case["sizes"].split(",")]
        state["sol"] = fm.Batch(case["kind"], sizes, case["h"], alpha=case["alpha"], **opts)
        total = sum(n * n for n in sizes)
        flat = [torch.empty(total, dtype=torch.float64, device="cuda") for _ in range(3)]
        views, at = [], 0
        for n in sizes:
            views.append([f[at:at + n * n].view(n, n) for f in flat])
            at += n * n
        state.update(out=flat, views=views, dts=[d[2] for d in data])
        return state
    if case["model"] == "gradflow":
        opts["model"] = fm.FM_GRADFLOW
    elif case.get("walls") is not None:
        opts.update(walls=fm.FM_WALLS_Y, u_wall=(-case["walls"], case["walls"]))
    elif case["extrapolate"]:
        opts["init"] = fm.FM_INIT_EXTRAPOLATE
    state["sol"] = fm.Solver(case["kind"], _ns(case), case["h"], dim=case["dim"], alpha=case.get("alpha", 0.0),
                             nu=case.get("nu", 0.0), delta=case.get("delta", 0.0), **opts)
    rho, vel, _ = data[0]
    state["out"] = [torch.empty_like(rho)] + [torch.empty_like(v) for v in vel]
    return state


def run(state):
    case, sol = state["case"], state["sol"]
    if case["model"] == "batch":
        for i, (rho, vel, _) in enumerate(state["data"]):
            sol.set_fields(i, rho, vel)
        for _ in range(case["steps"]):
            sol.step(state["dts"])
        for i, v in enumerate(state["views"]):
            fm.fm_get_fields(sol.instance(i), v[0], v[1:])
        return {"rho": state["out"][0], "vel": state["out"][1:]}
    rho, vel, dt = state["data"][0]
    flow = case["model"] == "gradflow"
    sol.set_fields(rho, None if flow else vel)
    terms = []
    for _ in range(case["steps"]):
        sol.step(dt)
        if case.get("energy"):
            terms.append(sol.energy_terms())
    out = state["out"]
    sol.get_fields(out[0], out[1:])
    res = {"rho": out[0], "vel": [] if flow else out[1:]}
    if terms:
        res["energy"] = torch.tensor(terms, dtype=torch.float64)
    return res


def work(case):
    """Bytes: the fields in and out, once.  Operations: per point and step, the
    source, closure and two residuals of a step, and one V(2, 2) cycle (four
    sweeps and a residual, times the sum of the coarser levels), counted from
    the equations; a step needs at least one cycle."""
    if case["model"] == "batch":
        pts, dim = sum(int(n) ** 2 for n in case["sizes"].split(",")), 2
    else:
        pts, dim = math.prod(_ns(case)), case["dim"]
    levels = 4.0 / 3.0 if dim == 2 else 8.0 / 7.0
    if case["model"] == "gradflow":
        per, fields = 20 + 2 * 30 + levels * (4 * 35 + 30), 1
    elif case["kind"] == "cdft":
        per, fields = 60 + 2 * 60 + levels * (4 * 80 + 60), 1 + dim
    else:
        per, fields = 45 * dim + 2 * 35 * dim + levels * (4 * 50 * dim + 35 * dim), 1 + dim
    return {"bytes": 16.0 * fields * pts, "flops": float(per) * pts * case["steps"]}


# --------------------------------------------------------------------------
# the same steps in float64 torch
# --------------------------------------------------------------------------
class _Grid:
    """Shifts, differences and the Laplacian, periodic or between walls in y.
    A field's `odd` says its ghost beyond a wall: None mirrors, a pair (bottom,
    top) gives 2 U - x."""

    def __init__(self, dim, h, walls):
        self.dim, self.h, self.walls = dim, h, walls

    def sh(self, a, d, k, odd=None):
        ax = a.dim() - 1 - d
        b = torch.roll(a, -k, ax)
        if self.walls is not None and d == 1:
            row = a.shape[ax] - 1 if k > 0 else 0
            edge = a.select(ax, row)
            if odd is not None:
                edge = 2.0 * odd[1 if k > 0 else 0] - edge
            b.select(ax, row).copy_(edge)
        return b

    def ghosts(self, a):
        """Ghost rule of velocity component a."""
        if self.walls is None:
            return None
        return (-self.walls, self.walls) if a == 0 else (0.0, 0.0)

    def D0(self, a, d, odd=None):
        return (self.sh(a, d, 1, odd) - self.sh(a, d, -1, odd)) / (2.0 * self.h)

    def lap(self, a, odd=None):
        acc = -2.0 * self.dim * a
        for d in range(self.dim):
            acc = acc + self.sh(a, d, 1, odd) + self.sh(a, d, -1, odd)
        return acc / (self.h * self.h)

    def div(self, rk, vel):
        acc = 0.0
        for d in range(self.dim):
            o = self.ghosts(d)
            acc = acc + (self.sh(rk, d, 1) * self.sh(vel[d], d, 1, o) - self.sh(rk, d, -1) * self.sh(vel[d], d, -1, o))
        return acc / (2.0 * self.h)

    def cross(self, om, U):
        if self.dim == 2:
            return [-om[0] * U[1], om[0] * U[0]]
        return [om[1] * U[2] - om[2] * U[1], om[2] * U[0] - om[0] * U[2], om[0] * U[1] - om[1] * U[0]]

    def curl(self, v):
        g = self.ghosts
        if self.dim == 2:
            return [self.D0(v[1], 0, g(1)) - self.D0(v[0], 1, g(0))]
        return [self.D0(v[2], 1) - self.D0(v[1], 2), self.D0(v[0], 2) - self.D0(v[2], 0),
                self.D0(v[1], 0) - self.D0(v[0], 1)]

    def grad_q(self, U):
        """Differences of |U|^2, the ghosts taken of its factors."""
        out = []
        for d in range(self.dim):
            p = sum(self.sh(U[c], d, 1, self.ghosts(c)) ** 2 for c in range(self.dim))
            m = sum(self.sh(U[c], d, -1, self.ghosts(c)) ** 2 for c in range(self.dim))
            out.append((p - m) / (2.0 * self.h))
        return out


def _kernel(ns, h, nu, dev):
    r2 = 0.0
    for d, n in enumerate(ns):
        k = _axis(n, d, len(ns), dev)
        r2 = r2 + (h * torch.minimum(k, n - k)) ** 2
    J = math.sqrt(2.0) * torch.exp(-math.pi ** 2 * r2 / (2 * nu * nu)) - torch.exp(-math.pi ** 2 * r2 / (4 * nu * nu))
    ce = float(torch.where(J <= 0, -J, torch.zeros_like(J)).sum()) * h ** len(ns)
    return torch.fft.fftn(J), ce


def _solve_mean(case, G, rk, s, ce, R):
    """A0^-1 R for the velocity residual R, A0 the momentum operator linearised
    about a uniform state of density rho0 (the middle of rk's range) at rest,
    the density and the chemical potential eliminated: in Fourier space
    (rho0 + s gamma lam / 2) I + (s rho0)^2 / 2 m k k^T, a rank-one update."""
    r0 = 0.5 * float(rk.max() + rk.min())
    lam, ks = 0.0, []
    for d in range(G.dim):
        n = rk.shape[G.dim - 1 - d]
        t = 2.0 * math.pi * _axis(n, d, G.dim, rk.device) / n
        lam = lam + (2.0 - 2.0 * torch.cos(t)) / (G.h * G.h)
        ks.append(torch.sin(t) / G.h)
    m = (r0 - 1.5) ** 2 + case["alpha"] + lam * lam if case["kind"] == "pfc" else 1.0 / r0 + 2.0 * ce
    a = r0 + 0.5 * s * GAMMA * lam
    b = 0.5 * (s * r0) ** 2 * m
    F = [torch.fft.fftn(r) for r in R]
    kf = sum(k * f for k, f in zip(ks, F)) * b / (a + b * sum(k * k for k in ks))
    return [torch.fft.ifftn((f - k * kf) / a).real for k, f in zip(ks, F)]


def _hydro_step(case, G, rk, uk, s, conv, ce):
    dim, h, pfc = G.dim, G.h, case["kind"] == "pfc"
    delta, gam = case.get("delta", 0.0), GAMMA
    om = G.curl(uk)
    wk = G.cross(om, uk)
    gh = G.ghosts
    S0 = rk - 0.5 * s * G.div(rk, uk)
    Su = [rk * (uk[a] - 0.5 * s * wk[a]) + 0.5 * s * gam * G.lap(uk[a], gh(a)) for a in range(dim)]
    if pfc:
        Smu = 2.0 * G.lap(rk)
    else:
        E = 2.0 * ce * rk + conv(rk)
        Su = [Su[a] + s * rk * G.D0(E, a) for a in range(dim)]
    diag = rk + s * gam * dim / (h * h)
    U = [u.clone() for u in uk]
    scale = max(float(u.abs().max()) for u in U) + 1e-3
    last = math.inf
    for it in range(6000):
        rho = S0 - 0.5 * s * G.div(rk, U)
        rho = torch.sqrt(rho * rho + delta * delta) if delta > 0 else rho.abs()
        if pfc:
            psi = rho - 1.5
            m = psi ** 3 / 3.0 + case["alpha"] * psi + G.lap(G.lap(rho)) + Smu
        else:
            m = torch.log(rho) + 2.0 * ce * rho
        gq = G.grad_q(U)
        wx = G.cross(om, U)
        R = [Su[a] - s * rk * (0.5 * wx[a] + 0.5 * gq[a] + G.D0(m, a)) + 0.5 * s * gam * G.lap(U[a], gh(a)) - rk * U[a]
             for a in range(dim)]
        if G.walls is None:
            R = _solve_mean(case, G, rk, s, ce, R)
        else:
            R = [r / diag for r in R]
        new = [U[a] + R[a] for a in range(dim)]
        if it % 8 == 7:
            change = max(float((new[a] - U[a]).abs().max()) for a in range(dim)) / scale
            U = new
            if change < 1e-15 or (change < 1e-13 and change >= last):
                break
            last = change
        else:
            U = new
    rho = S0 - 0.5 * s * G.div(rk, U)
    return (torch.sqrt(rho * rho + delta * delta) if delta > 0 else rho.abs()), U


def _flow_step(case, G, rk, s):
    lam = 0.0
    for d in range(G.dim):
        n = rk.shape[G.dim - 1 - d]
        lam = lam + (2.0 - 2.0 * torch.cos(2.0 * math.pi * _axis(n, d, G.dim, rk.device) / n)) / (G.h * G.h)
    Smu = 2.0 * G.lap(rk)
    rho, last = rk.clone(), math.inf
    for _ in range(400):
        psi = rho - 1.5
        mu = psi ** 3 / 3.0 + case["alpha"] * psi + G.lap(G.lap(rho)) + Smu
        F = rho - s * G.lap(mu) - rk
        qb = float((psi * psi).mean()) + case["alpha"]
        d = torch.fft.ifftn(torch.fft.fftn(F) / (1.0 + s * lam * (qb + lam * lam))).real
        rho = rho - d
        change = float(d.abs().max())
        if change < 1e-15 or (change < 1e-12 and change >= 0.5 * last):
            break
        last = change
    psi = rho - 1.5
    mu = psi ** 3 / 3.0 + case["alpha"] * psi + G.lap(G.lap(rho)) + Smu
    return (rk + s * G.lap(mu)).abs()


def _energy(case, G, rho, vel, conv):
    w = G.h ** G.dim
    KE = 0.5 * w * float((rho * sum(v * v for v in vel)).sum())
    if case["kind"] == "cdft":
        return [KE, w * float((rho * (torch.log(rho) - 1.0)).sum()), -0.5 * w * float((rho * conv(rho)).sum()), 0.0, 0.0]
    psi, L = rho - 1.5, G.lap(rho)
    return [KE, w * float((psi ** 4).sum()) / 12.0, 0.5 * w * case["alpha"] * float((psi ** 2).sum()),
            0.5 * w * float((L * L).sum()), w * float((rho * L).sum())]


def exact(case, seed):
    """run()'s outputs for the same inputs: the scheme's steps solved in
    float64 by fixed-point iteration on the velocity (the density and chemical
    potential eliminated), preconditioned by the operator of a uniform state
    (periodic) or its diagonal (walls)."""
    data = _inputs(case, seed)
    rhos, vels, energies = [], [[] for _ in range(case["dim"])], []
    for rho, vel, dt in data:
        G = _Grid(case["dim"], case["h"], case.get("walls"))
        conv, ce = None, 0.0
        if case["kind"] == "cdft":
            Jh, ce = _kernel(_ns(case), case["h"], case["nu"], rho.device)
            w = case["h"] ** case["dim"]
            conv = lambda x: w * torch.fft.ifftn(Jh * torch.fft.fftn(x)).real  # noqa: E731
        for _ in range(case["steps"]):
            if case["model"] == "gradflow":
                rho = _flow_step(case, G, rho, dt)
            else:
                rho, vel = _hydro_step(case, G, rho, vel, dt, conv, ce)
            if case.get("energy"):
                energies.append(_energy(case, G, rho, vel, conv))
        rhos.append(rho)
        for a in range(case["dim"]):
            vels[a].append(vel[a])
    if case["model"] == "batch":
        return {"rho": torch.cat([r.reshape(-1) for r in rhos]), "vel": [torch.cat([v.reshape(-1) for v in c]) for c in vels]}
    res = {"rho": rhos[0], "vel": [] if case["model"] == "gradflow" else [c[0] for c in vels]}
    if energies:
        res["energy"] = torch.tensor(energies, dtype=torch.float64)
    return res
