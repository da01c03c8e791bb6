"""The float64 V-cycle of the coarsest levels by a cluster of blocks
(fm_cluster.cuh), every component at every point: the iterate left by one damped
cycle against the oracle's cycle, with clusters of 16 blocks and of 8 (FM_CLUSTER=8,
the size where 16 cannot be scheduled), on velocities for which the vorticity and
kinetic terms are of the size of the others.

The oracle linearises the cubic of the mu row about the current density, the
library evaluates it at the new one; the oracle's update is corrected by that
(`_exact_cubic`).  Tolerances, derived before the first run, relative to the
row's largest correction: float64 rounds a few dozen updates whose rows are scaled
by up to 4 d / h^2 ~ 15, below 1e-12, bound 1e-10; the mixed path rounds the
cycle's data and corrections to 6e-8 besides, below 1e-5 after the same scaling
twice, bound 1e-4.  Dropping the vorticity or the kinetic term, or transposing the 3-D
velocity block, in the oracle's update changes some row by 2e-3 or more
(test_the_bounds_reject_mistakes)."""
import numpy as np
import pytest

from oracle import scheme as S
from paper_1503_07416_gb300 import fm

# the largest and smallest levels, long rows and columns, levels whose points do
# not fill the last block, 3-D (16 x 16 x 4: the largest shared memory)
GRIDS = [("pfc", (32, 32)), ("pfc", (30, 34)), ("pfc", (512, 2)), ("pfc", (2, 512)), ("pfc", (6, 4)), ("pfc", (2, 2)),
         ("pfc", (16, 16, 4)), ("pfc", (8, 10, 12)), ("cdft", (32, 32)), ("cdft", (64, 4)), ("cdft", (8, 8, 16))]
OPTS = S.SolverOpts(nu1=1, nu2=1, coarsest=2, ncoarse=2)


def _problem(kind, n):
    rng = np.random.default_rng(31)
    shape = tuple(reversed(n))
    if kind == "pfc":
        rho = 0.8 + 0.05 * rng.uniform(-1, 1, shape)
        P, J = S.Params(kind=S.PFC, dim=len(n), h=0.9, s=0.4, gamma=0.1, alpha=0.6, w_damp=0.5), None
        vel = [0.5 * rng.standard_normal(shape) for _ in n]
    else:
        rho = 0.3 + 0.03 * rng.uniform(-1, 1, shape)
        J, ce = S.cdft_setup(shape, 0.5, 2.362)
        P = S.Params(kind=S.CDFT, dim=len(n), h=0.5, s=0.1, gamma=0.1, ce=ce, delta=1e-10, w_damp=0.5)
        vel = [0.2 * rng.standard_normal(shape) for _ in n]
    return rho, vel, P, J


def _exact_cubic(update):
    """The oracle's point update with mu's cubic at the new density."""
    def point_update(g, f, c, P, mask):
        old = g[0].copy()
        update(g, f, c, P, mask)
        if P.kind == S.PFC:
            p0 = old - 1.5
            p1 = (g[0] - P.w_damp * old) / (1.0 - P.w_damp) - 1.5  # before the damping
            g[1 + P.dim] = np.where(mask, g[1 + P.dim] + (1.0 - P.w_damp) * (p1 ** 3 / 3.0 - (p0 ** 2 * p1 - p0 ** 3 * 2 / 3)),
                                    g[1 + P.dim])
    return point_update


def _oracle_correction(kind, n, monkeypatch, mistake=None):
    rho, vel, P, J = _problem(kind, n)
    c = S.Coeffs(rho, S.vorticity(vel, P.h))
    f = S.source(rho, vel, c.om, P, S.conv_fft(J, rho, P.h) if J is not None else None)
    g0 = S.initial_iterate(rho, vel, P)
    g = [x.copy() for x in g0]
    update = S.point_update

    def with_mistake(g, f, c, P, mask):
        if mistake == "omega":
            c = S.Coeffs(c.rk, [0.0 * w for w in c.om])
        if mistake == "transpose":
            c = S.Coeffs(c.rk, [-w for w in c.om])
        if mistake == "kinetic":
            f = list(f)
            q = sum(g[1 + a] ** 2 for a in range(P.dim))
            for a in range(P.dim):
                f[1 + a] = f[1 + a] + 0.5 * P.s * c.rk * S.D0(q, a, P.h)
        update(g, f, c, P, mask)

    with monkeypatch.context() as m:
        m.setattr(S, "point_update", _exact_cubic(with_mistake))
        S.vcycle(g, f, c, P, OPTS)
    return [a - b for a, b in zip(g, g0)]


@pytest.mark.parametrize("mistake", ["omega", "kinetic", "transpose"])
@pytest.mark.parametrize("kind,n", [g for g in GRIDS if g[1] not in ((512, 2), (2, 512), (2, 2))])
def test_the_bounds_reject_mistakes(kind, n, mistake, monkeypatch):
    want = _oracle_correction(kind, n, monkeypatch)
    wrong = _oracle_correction(kind, n, monkeypatch, mistake)
    assert max(np.max(np.abs(a - b)) / np.max(np.abs(b)) for a, b in zip(wrong, want)) >= 2e-3


@pytest.mark.gpu
@pytest.mark.parametrize("blocks", [16, 8])
@pytest.mark.parametrize("precision", [fm.FM_FP64, fm.FM_MIXED])
@pytest.mark.parametrize("kind,n", GRIDS)
def test_cluster_cycle_rows(kind, n, precision, blocks, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rho, vel, P, _ = _problem(kind, n)
    kw = dict(alpha=0.6) if kind == "pfc" else dict(nu=2.362, delta=1e-10)
    if blocks == 8:
        monkeypatch.setenv("FM_CLUSTER", "8")
    sol = fm.Solver(kind, n, P.h, dim=P.dim, precision=precision, gamma=P.gamma, w_damp=P.w_damp, nu1=1, nu2=1, ncoarse=2,
                    coarsest=2, tol=1e-300, max_cycles=1, **kw)
    assert fm.fm_cluster_blocks(sol.handle) == blocks
    sol.set_fields(rho, vel)
    fm.fm_prepare(sol.handle, P.s)
    g0 = [sol.aux(fm.FM_AUX_ITERATE, q) for q in range(sol.nu)]
    code, info = fm.fm_step_raw(sol.handle, P.s)
    assert code == fm.FM_ENOCONV and info.cycles == 1
    e = [sol.aux(fm.FM_AUX_ITERATE, q) - g0[q] for q in range(sol.nu)]
    sol.close()
    bound = 1e-10 if precision == fm.FM_FP64 else 1e-4
    for q, (a, b) in enumerate(zip(e, _oracle_correction(kind, n, monkeypatch))):
        size = np.max(np.abs(b)) or np.max(np.abs(g0[q]))  # (2 x 2: every difference and mu's correction are 0)
        assert np.max(np.abs(a - b)) <= bound * size, q
