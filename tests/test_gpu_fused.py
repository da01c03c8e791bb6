"""The fused 2-D level kernels of the gradient flow and the channel
(fm_fused.cuh): the residual left by one damped V(nu1, nu2) cycle against the
oracle's cycle on the same state.

Tolerances, derived before the first run.  Gradient flow: the oracle and the
library run the same point block, so float64 agrees to rounding, far below
1e-7; float32 rounds corrections and coefficients to 6e-8 in a few dozen
updates of a system whose rows are scaled by up to 2 d / h^2 ~ 5, so the
residual, of the order of the first one after a damped cycle, agrees to
1e-4.  Channel: the oracle's cycle with the library's point block (below); the
oracle linearises the cubic about the current density, the library evaluates
it at the new one, which differ by ~1e-5 of the change here: 1e-3 for both
precisions.  A wrong neighbour, ghost, tile edge or skipped sweep shows at the
percent level."""
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


# (nx, ny): both tile sizes with a ragged last tile, rows that are no whole
# number of 16 bytes, levels of the one-block part only, a tile wider than the
# grid; (nu1, nu2): two sweeps a launch, an odd last sweep, none
GRIDS = [((272, 136), (2, 2)), ((66, 40), (2, 2)), ((44, 52), (1, 2)), ((36, 20), (2, 2)), ((8, 260), (3, 1)),
         ((128, 72), (0, 2))]


def _residual_after_one_cycle(sol, s):
    code, info = fm.fm_step_raw(sol.handle, s)
    sol.close()
    assert code == fm.FM_ENOCONV and info.cycles == 1
    return info.res


@pytest.mark.parametrize("precision", [fm.FM_FP64, fm.FM_MIXED])
@pytest.mark.parametrize("n,nu", GRIDS)
@pytest.mark.parametrize("kind", ["pfc", "cdft"])
def test_gradflow_cycle_equals_oracle(kind, n, nu, precision):
    if kind == "cdft":
        n = tuple(1 << (k - 1).bit_length() for k in n)  # the convolution wants powers of two
    rng = np.random.default_rng(3)
    shape = (n[1], n[0])
    if kind == "pfc":
        rho = 0.8 + 0.05 * rng.uniform(-1, 1, shape)
        P, J, extra = S.Params(kind=S.PFC, dim=2, h=0.9, s=0.02, alpha=0.6, w_damp=0.5), None, dict(alpha=0.6)
    else:
        rho = 0.3 + 0.03 * rng.uniform(0, 1, shape)
        J, ce = S.cdft_setup(shape, 0.5, 2.362)
        P = S.Params(kind=S.CDFT, dim=2, h=0.5, s=0.02, ce=ce, delta=1e-10, w_damp=0.5)
        extra = dict(nu=2.362, delta=1e-10)
    opts = S.SolverOpts(nu1=nu[0], nu2=nu[1], coarsest=4, ncoarse=3)
    f = GF.source(rho, P, S.conv_fft(J, rho, P.h) if J is not None else None)
    g = GF.initial_iterate(rho, P)
    GF.vcycle(g, f, P, opts)
    want = S.res_norm(GF.residual(g, f, P), P.h)
    sol = fm.Solver(kind, n, P.h, model=fm.FM_GRADFLOW, precision=precision, w_damp=0.5, nu1=nu[0], nu2=nu[1], coarsest=4,
                    ncoarse=3, tol=1e-300, max_cycles=1, **extra)
    sol.set_fields(rho, None)
    got = _residual_after_one_cycle(sol, P.s)
    assert abs(got - want) <= (1e-7 if precision == fm.FM_FP64 else 1e-4) * want, (got, want)


def _lagged_ghost_update(g, f, c, P, W, mask):
    """The channel's point block with the ghosts of a wall row taken from its
    values before the update, as the library does.  (The oracle's own block
    moves a wall row's ghost, which mirrors the row itself, to the left side;
    the same fixed point, another iterate at the wall rows.)"""
    h, s, w, rk = P.h, P.s, P.w_damp, c.rk
    old = [x.copy() for x in g]
    rho = np.abs(f[0] - 0.5 * s * Ch.div_rk(rk, [old[1], old[2]], h, W))
    kap = f[4] + (Ch.nb_sum(old[0], Ch.SCAL, W) - 4.0 * rho) / (h * h)
    psi = rho - 1.5
    mu = f[3] + psi ** 3 / 3.0 + P.alpha * psi + (Ch.nb_sum(old[4], Ch.SCAL, W) - 4.0 * kap) / (h * h)
    rhs = [f[1 + a] + s * (-0.5 * rk * Ch.D0q([old[1], old[2]], a, h, W) - rk * Ch.D0(old[3], a, h, Ch.SCAL, W)
                           + 0.5 * P.gamma * Ch.nb_sum(old[1 + a], Ch.VEL_T[a], W) / (h * h)) for a in range(2)]
    A, b = rk + 2.0 * s * P.gamma / (h * h), 0.5 * P.sigma * s * rk * c.om[0]
    new = [rho, (A * rhs[0] + b * rhs[1]) / (A * A + b * b), (A * rhs[1] - b * rhs[0]) / (A * A + b * b), mu, kap]
    for i in range(5):
        g[i] = np.where(mask, (1.0 - w) * new[i] + w * old[i], old[i])


@pytest.mark.parametrize("precision", [fm.FM_FP64, fm.FM_MIXED])
@pytest.mark.parametrize("n,nu", GRIDS)
def test_channel_cycle_equals_oracle(n, nu, precision, monkeypatch):
    monkeypatch.setattr(Ch, "point_update", _lagged_ghost_update)
    rng = np.random.default_rng(4)
    shape = (n[1], n[0])
    rho = 0.8 + 0.05 * rng.uniform(-1, 1, shape)
    vel = [1e-3 * rng.standard_normal(shape) for _ in range(2)]
    P = S.Params(kind=S.PFC, dim=2, h=0.9, s=0.02, alpha=0.6, w_damp=0.5)
    W = Ch.Walls(-2e-3, 1e-3)
    opts = S.SolverOpts(nu1=nu[0], nu2=nu[1], coarsest=4, ncoarse=3)
    c = Ch.Coeffs(rho, Ch.vorticity(vel, P.h, W))
    f = Ch.source(rho, vel, c.om, P, W)
    g = Ch.initial_iterate(rho, vel, P, W)
    Ch.vcycle(g, f, c, P, W, opts)
    want = S.res_norm(Ch.residual(g, f, c, P, W), P.h)
    sol = fm.Solver("pfc", n, P.h, alpha=0.6, precision=precision, w_damp=0.5, nu1=nu[0], nu2=nu[1], coarsest=4, ncoarse=3,
                    tol=1e-300, max_cycles=1, walls=fm.FM_WALLS_Y, u_wall=(-2e-3, 1e-3))
    sol.set_fields(rho, vel)
    got = _residual_after_one_cycle(sol, P.s)
    assert abs(got - want) <= 1e-3 * want, (got, want)
