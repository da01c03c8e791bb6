"""The float64 source and residual keep float64's relative accuracy where the
fields are small beside larger ones: a loud patch in a quiet field (velocity,
density, mu and kappa 1e-9 of the patch's) and a velocity component far weaker
than the others, every point compared at its own size.

Reference: the rows in extended precision (numpy's long double), each value with
the sum m of the magnitudes of the terms it is made of at that point.
Tolerance, derived before the first run: a row takes at most 14 roundings on the
way from the inputs (the vorticity's 4, a coefficient's 2, a product's, a
difference's and the chain's), each of at most 2^-53 of the terms at that
point: 16 x 2^-53 m.  A sum whose values are held relative to something larger
than the point's own terms exceeds it by the ratio of the two."""
import numpy as np
import pytest

from oracle import channel as Ch
from oracle import gradflow as GF
from oracle import scheme as S
from paper_1503_07416_gb300 import fm

pytestmark = pytest.mark.gpu
LD = np.longdouble
U_BOT, U_TOP = -3e-9, 2e-9  # quiet walls


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_07416_gb300 import build
    build.build_library()
    fm.lib()


class V:
    """A value in extended precision and the sum of its terms' magnitudes."""

    def __init__(self, v, m=None):
        self.v = np.asarray(v, LD)
        self.m = np.abs(self.v) if m is None else m

    def __add__(self, o):
        o = o if isinstance(o, V) else V(o)
        return V(self.v + o.v, self.m + o.m)

    def __sub__(self, o):
        o = o if isinstance(o, V) else V(o)
        return V(self.v - o.v, self.m + o.m)

    def __mul__(self, o):
        o = o if isinstance(o, V) else V(o)
        return V(self.v * o.v, self.m * o.m)

    __radd__, __rmul__ = __add__, __mul__


class Ops:
    def __init__(self, dim, h, walls):
        self.dim, self.h, self.walls = dim, LD(h), walls

    def sh(self, a, d, k, comp=None):
        """a one point along d; comp: the velocity component (its ghost beyond a wall)."""
        ax = self.dim - 1 - d
        b = V(np.roll(a.v, -k, ax), np.roll(a.m, -k, ax))
        if self.walls and d == 1:
            row = -1 if k > 0 else 0
            U = LD(U_TOP if k > 0 else U_BOT) if comp == 0 else LD(0)
            if comp is None:
                b.v[row], b.m[row] = a.v[row], a.m[row]
            else:
                b.v[row], b.m[row] = 2 * U - a.v[row], 2 * abs(U) + a.m[row]
        return b

    def diff(self, f, d):
        """f(k) at +1 less f(k) at -1, f(k) shifted by k along d."""
        return f(d, 1) - f(d, -1)

    def lap(self, a, comp=None):
        acc = V(LD(-2 * self.dim)) * a
        for d in range(self.dim):
            acc = acc + self.sh(a, d, 1, comp) + self.sh(a, d, -1, comp)
        return acc * (1 / (self.h * self.h))

    def div(self, rk, u):
        """div_h(rho^k u)."""
        return sum((self.diff(lambda d, k: self.sh(rk, d, k) * self.sh(u[d], d, k, d), d) for d in range(self.dim)),
                   V(LD(0))) * (1 / (2 * self.h))

    def grad(self, f, d):
        return self.diff(f, d) * (1 / (2 * self.h))

    def curl(self, u):
        D = lambda c, d: self.grad(lambda e, k: self.sh(u[c], e, k, c), d)  # noqa: E731
        if self.dim == 2:
            return [D(1, 0) - D(0, 1)]
        return [D(2, 1) - D(1, 2), D(0, 2) - D(2, 0), D(1, 0) - D(0, 1)]

    def cross(self, om, u):
        if self.dim == 2:
            return [V(LD(-1)) * om[0] * u[1], om[0] * u[0]]
        return [om[(a + 1) % 3] * u[(a + 2) % 3] - om[(a + 2) % 3] * u[(a + 1) % 3] for a in range(3)]


CASES = [("pfc", (36, 20), m) for m in ("periodic", "walls", "gradflow")]
CASES += [("pfc", (130, 72), m) for m in ("periodic", "walls", "gradflow")]
CASES += [("cdft", (64, 32), "periodic"), ("pfc", (10, 6, 14), "periodic"), ("pfc", (10, 6, 14), "gradflow"),
          ("cdft", (16, 8, 32), "periodic")]


@pytest.mark.parametrize("kind,n,model", CASES)
def test_rows_are_accurate_at_every_point(kind, n, model):
    rng = np.random.default_rng(21)
    shape, dim, h, s, gamma = tuple(reversed(n)), len(n), 0.75, 0.03125, 2.0
    loud = np.full(shape, 1e-9)
    loud[tuple(slice(k // 2, k // 2 + 4) for k in shape)] = 1.0
    field = lambda a, b: loud * (a + b * rng.uniform(-1, 1, shape))  # noqa: E731
    rho = field(0.8, 0.05)
    vel = [(1e-5 if a == 1 else 0.1) * loud * rng.standard_normal(shape) for a in range(dim)]
    flow = model == "gradflow"
    extra, ce = dict(alpha=0.6) if kind == "pfc" else dict(nu=2.362, delta=0.0), 0.0
    if kind == "cdft":
        ce = S.cdft_setup(shape, h, 2.362)[1]
    if flow:
        extra["model"] = fm.FM_GRADFLOW
    if model == "walls":
        extra.update(walls=fm.FM_WALLS_Y, u_wall=(U_BOT, U_TOP))
    sol = fm.Solver(kind, n, h, dim=dim, precision=fm.FM_FP64, gamma=gamma, **extra)
    sol.set_fields(rho, None if flow else vel)
    fm.fm_prepare(sol.handle, s)
    nom = 0 if flow else (1 if dim == 2 else 3)
    om = [sol.aux(fm.FM_AUX_OMEGA, c) for c in range(nom)]
    src = [sol.aux(fm.FM_AUX_SOURCE, c) for c in range(sol.nu)]
    g0 = [sol.aux(fm.FM_AUX_ITERATE, c) for c in range(sol.nu)]
    conv = sol.aux(fm.FM_AUX_CONV, 0) if kind == "cdft" else None
    g = [field(0.8, 0.05)] + ([] if flow else [(1e-5 if a == 1 else 0.1) * loud * rng.standard_normal(shape) for a in range(dim)])
    g += [loud * rng.standard_normal(shape) for _ in range(sol.nu - len(g))]
    r = [np.empty(shape) for _ in g]
    fm.fm_residual(sol.handle, g, r)
    sol.close()

    O, rk, s_ = Ops(dim, h, model == "walls"), V(rho), LD(s)
    checks = []  # (what, got, want)
    G, src_v = [V(x) for x in g], [V(x) for x in src]
    psi = G[0] - LD(1.5)
    mu_row = lambda m, k: m - psi * psi * psi * (LD(1) / 3) - psi * LD(0.6) - O.lap(k)  # noqa: E731
    if flow:
        checks += [("S_mu", src[1], O.lap(rk) * LD(2)), ("kappa0", g0[2], O.lap(rk))]
        checks += [("r0", r[0], src_v[0] - (G[0] - O.lap(G[1]) * s_)), ("r1", r[1], src_v[1] - mu_row(G[1], G[2])),
                   ("r2", r[2], O.lap(G[0]) - G[2])]
    else:
        u = [V(x) for x in vel]
        w = O.curl(u)
        checks += [(f"omega{c}", om[c], w[c]) for c in range(nom)]
        checks.append(("S0", src[0], rk - O.div(rk, u) * (s_ / 2)))
        wx = O.cross(w, u)
        for a in range(dim):
            row = rk * (u[a] - wx[a] * (s_ / 2)) + O.lap(u[a], a) * (s_ * LD(gamma) / 2)
            if kind == "cdft":
                E = rk * LD(2 * ce) + V(conv)
                row = row + rk * O.grad(lambda d, k: O.sh(E, d, k), a) * s_
            checks.append((f"S{1 + a}", src[1 + a], row))
        u, om_v = G[1:1 + dim], [V(x) for x in om]
        if kind == "pfc":
            checks += [("S_mu", src[1 + dim], O.lap(rk) * LD(2)), ("kappa0", g0[2 + dim], O.lap(rk))]
            m = G[1 + dim]
            checks += [("r_mu", r[1 + dim], src_v[1 + dim] - mu_row(m, G[2 + dim])), ("r_kappa", r[2 + dim], O.lap(G[0]) - G[2 + dim])]
        else:
            m = V(np.log(G[0].v)) + G[0] * LD(2 * ce)
        checks.append(("r0", r[0], src_v[0] - (G[0] + O.div(rk, u) * (s_ / 2))))
        wx = O.cross(om_v, u)
        for a in range(dim):
            q = lambda d, k: sum((O.sh(u[c], d, k, c) * O.sh(u[c], d, k, c) for c in range(dim)), V(LD(0)))  # noqa: E731
            br = u[a] + wx[a] * (s_ / 2) + O.grad(q, a) * (s_ / 2) + O.grad(lambda d, k: O.sh(m, d, k), a) * s_
            checks.append((f"r{1 + a}", r[1 + a], src_v[1 + a] - rk * br + O.lap(u[a], a) * (s_ * LD(gamma) / 2)))
    tol = LD(16) * LD(2) ** -53
    for what, got, want in checks:
        err = np.abs(got.astype(LD) - want.v) / (want.m + LD(1e-300))
        assert np.max(err) <= tol, (what, float(np.max(err) / tol), int(np.sum(err > tol)))


@pytest.mark.parametrize("value", [1e305, np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("n,model", [((36, 20), "periodic"), ((36, 20), "walls"), ((36, 20), "gradflow"),
                                     ((10, 6, 14), "periodic"), ((10, 6, 14), "gradflow")])
def test_values_beyond_fixed_point(n, model, value):
    """A kappa (and, finite, a velocity) that the fixed-point sums do not take:
    the rows are the float64 ones, points beside it to rounding (1e-12 of the
    larger of 1 and the row's largest ordinary or huge value), the others as if it
    were not there, non-finite where the float64 sums are."""
    rng = np.random.default_rng(22)
    shape, dim, h, s = tuple(reversed(n)), len(n), 0.7, 0.03
    rho = 0.8 + 0.05 * rng.uniform(-1, 1, shape)
    vel = [0.1 * rng.standard_normal(shape) for _ in n]
    P = S.Params(kind=S.PFC, dim=dim, h=h, s=s, alpha=0.6)
    W, extra = Ch.Walls(-0.2, 0.1), dict(alpha=0.6)
    at = rho.size // 3
    if model == "gradflow":
        extra["model"] = fm.FM_GRADFLOW
    elif np.isfinite(value):
        vel[0].flat[at] = value
    if model == "walls":
        extra.update(walls=fm.FM_WALLS_Y, u_wall=(W.u_bot, W.u_top))
    sol = fm.Solver("pfc", n, h, dim=dim, precision=fm.FM_FP64, **extra)
    g = [rho] + ([] if model == "gradflow" else [0.1 * rng.standard_normal(shape) for _ in n])
    g += [rng.standard_normal(shape) for _ in range(2)]
    g[-1].flat[at] = value
    with np.errstate(all="ignore"):
        if model == "gradflow":
            f, want_s = GF.source(rho, P), []
            want_r = GF.residual(g, f, P)
        elif model == "walls":
            om = Ch.vorticity(vel, h, W)
            want_s = f = Ch.source(rho, vel, om, P, W)
            want_r = Ch.residual(g, f, Ch.Coeffs(rho, om), P, W)
        else:
            om = S.vorticity(vel, h)
            want_s = f = S.source(rho, vel, om, P, None)
            want_r = S.residual(g, f, S.Coeffs(rho, om), P)
        sol.set_fields(rho, None if model == "gradflow" else vel)
        fm.fm_prepare(sol.handle, s)
        got = [sol.aux(fm.FM_AUX_SOURCE, c) for c in range(len(want_s))]
        r = [np.empty(shape) for _ in g]
        fm.fm_residual(sol.handle, g, r)
        sol.close()
        for a, b in zip(got + r, list(want_s) + list(want_r)):
            for mask in (np.abs(b) < 1e100, (np.abs(b) >= 1e100) & np.isfinite(b)):
                if mask.any():
                    assert np.max(np.abs(a[mask] - b[mask])) <= 1e-12 * max(1.0, np.max(np.abs(b[mask])))
            assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isposinf(a), np.isposinf(b))
            assert np.array_equal(np.isneginf(a), np.isneginf(b))
