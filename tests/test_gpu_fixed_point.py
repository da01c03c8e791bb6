"""The float64 source and residual kernels whose neighbour sums run in fixed
point (to_fix in fm_device.cuh), and their float64 branch for values beyond its
range, against the oracle's omega, S, g^0 and S - N(g).

Tolerances, derived before the first run: a fixed-point value keeps at least
58 bits below the largest of its tile, so a row is off by less than float64's
own rounding of its largest term; 1e-12 of max(1, the row's largest value), as
for the residual rows elsewhere.  With one velocity of 1e130 the rows near it
are compared at their own size and all others at theirs, so that a neighbour
tile that left fixed point needlessly or not at all shows."""
import numpy as np
import pytest

from oracle import channel as Ch
from oracle import gradflow as GF
from oracle import scheme as S
from paper_1503_07416_gb300 import fm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_07416_gb300 import build
    build.build_library()
    fm.lib()


def _close(got, want):
    for big in (False, True):
        m = (np.abs(want) >= 1e100) == big
        if m.any():
            assert np.max(np.abs(got[m] - want[m])) <= 1e-12 * max(1.0, np.max(np.abs(want[m]))), big


# ragged and single tiles, grids narrower than a halo, several tiles; 3-D
# planes that do not fill the last block
GRIDS = [("pfc", (36, 20)), ("pfc", (2, 70)), ("pfc", (70, 2)), ("pfc", (130, 72)), ("pfc", (10, 6, 14)),
         ("pfc", (64, 4, 2)), ("cdft", (64, 32)), ("cdft", (16, 8, 32))]
CASES = [(k, n, m) for k, n in GRIDS for m in ("periodic", "walls", "gradflow") if m == "periodic" or len(n) == 2 and k == "pfc"]


@pytest.mark.parametrize("vel_of", ["ordinary", "zero", "spike"])
@pytest.mark.parametrize("kind,n,model", CASES)
def test_source_and_residual_rows(kind, n, model, vel_of):
    rng = np.random.default_rng(11)
    shape, dim, h, s = tuple(reversed(n)), len(n), 0.7, 0.03
    rho = (0.8 if kind == "pfc" else 0.3) + 0.05 * rng.uniform(-1, 1, shape)
    vel = [(0.0 if vel_of == "zero" else 0.1) * rng.standard_normal(shape) for _ in n]
    if vel_of == "spike":
        vel[0].flat[rho.size // 3] = 1e130
    if kind == "pfc":
        P, J, extra = S.Params(kind=S.PFC, dim=dim, h=h, s=s, alpha=0.6), None, dict(alpha=0.6)
    else:
        J, ce = S.cdft_setup(shape, h, 2.362)
        P, extra = S.Params(kind=S.CDFT, dim=dim, h=h, s=s, ce=ce, delta=1e-10), dict(nu=2.362, delta=1e-10)
    W, om = Ch.Walls(-0.2, 0.1), []
    if model == "gradflow":
        extra["model"], vel = fm.FM_GRADFLOW, []
        f, g0 = GF.source(rho, P), GF.initial_iterate(rho, P)
    elif model == "walls":
        extra.update(walls=fm.FM_WALLS_Y, u_wall=(W.u_bot, W.u_top))
        om = Ch.vorticity(vel, h, W)
        f, g0 = Ch.source(rho, vel, om, P, W), Ch.initial_iterate(rho, vel, P, W)
    else:
        om = S.vorticity(vel, h)
        f = S.source(rho, vel, om, P, S.conv_fft(J, rho, h) if J is not None else None)
        g0 = S.initial_iterate(rho, vel, P)
    sol = fm.Solver(kind, n, h, precision=fm.FM_FP64, **({"dim": dim} | extra))
    sol.set_fields(rho, vel or None)
    fm.fm_prepare(sol.handle, s)
    for what, rows in ((fm.FM_AUX_OMEGA, om), (fm.FM_AUX_SOURCE, f), (fm.FM_AUX_ITERATE, g0)):
        for c, want in enumerate(rows):
            _close(sol.aux(what, c), want)
    g = [rho + 0.01 * rng.standard_normal(shape)] + [v + 0.01 * rng.standard_normal(shape) for v in vel]
    g += [rng.standard_normal(shape) for _ in range(len(g0) - len(g))]
    if model == "gradflow" and vel_of == "spike":
        g[2].flat[rho.size // 3] = 1e130
    r = [np.empty(shape) for _ in g]
    fm.fm_residual(sol.handle, g, r)
    if model == "gradflow":
        want = GF.residual(g, f, P)
    elif model == "walls":
        want = Ch.residual(g, f, Ch.Coeffs(rho, om), P, W)
    else:
        want = S.residual(g, f, S.Coeffs(rho, om), P)
    sol.close()
    for a, b in zip(r, want):
        _close(a, b)
