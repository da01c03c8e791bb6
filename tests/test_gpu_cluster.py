"""The float64 coarse-grid kernels (fm_cluster.cuh: the cluster V-cycle of the
small levels, the tile sweeps of a larger 2-D coarsest level) against the
float32 ones, separate implementations of the same cycle: the residual left
by one damped cycle.

Tolerance, derived before the first run: the damped cycle leaves a residual of
the order of the first one (its factor is ~0.3), and the float32 cycle's
corrections and coefficients are rounded to 6e-8 relative in a few dozen
updates, so the two residuals agree to a few 1e-6 relative; a wrong neighbour,
ghost, transfer weight or skipped point changes them at the percent level.
Bound: 1e-4."""
import numpy as np
import pytest

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


# whole grids of at most 1,024 points: the largest and smallest levels, long
# rows and columns, levels whose points do not fill the last block, 3-D
GRIDS = [("pfc", (32, 32)), ("pfc", (30, 34)), ("pfc", (512, 2)), ("pfc", (2, 512)), ("pfc", (6, 4)), ("pfc", (2, 2)),
         ("pfc", (16, 16, 4)), ("pfc", (8, 10, 12)), ("cdft", (32, 32)), ("cdft", (64, 4)), ("cdft", (8, 8, 16))]


@pytest.mark.parametrize("kind,n", GRIDS)
@pytest.mark.parametrize("precision", [fm.FM_FP64, fm.FM_MIXED])
def test_cluster_cycle_equals_one_block_cycle(kind, n, precision):
    rng = np.random.default_rng(7)
    shape = tuple(reversed(n))
    rho = (0.8 if kind == "pfc" else 0.3) + 0.03 * rng.uniform(-1, 1, shape)
    vel = [0.05 * rng.standard_normal(shape) for _ in n]
    opts = dict(dim=len(n), w_damp=0.5, nu1=1, nu2=1, ncoarse=2, coarsest=2, tol=1e-300, max_cycles=1)
    opts.update(dict(alpha=0.6) if kind == "pfc" else dict(nu=2.362, delta=1e-10))
    res = []
    for prec, coarse in ((precision, fm.FM_FP64), (fm.FM_MIXED, fm.FM_MIXED)):
        sol = fm.Solver(kind, n, 0.9 if kind == "pfc" else 0.25, precision=prec, coarse_precision=coarse, **opts)
        sol.set_fields(rho, vel)
        code, info = fm.fm_step_raw(sol.handle, 0.02)
        assert code == fm.FM_ENOCONV and info.cycles == 1
        res.append((info.res0, info.res))
        sol.close()
    (a0, a), (b0, b) = res
    assert abs(a0 - b0) <= 1e-6 * b0
    assert abs(a - b) <= 1e-4 * b, (a, b)


# a coarsest level of more than 1,024 points that is the whole grid: ragged
# tiles, rows shorter than a tile's halo; odd sweep counts
TILES = [("pfc", (64, 64)), ("pfc", (90, 50)), ("pfc", (36, 38)), ("pfc", (4, 512)), ("pfc", (1024, 2)),
         ("cdft", (64, 64)), ("cdft", (128, 16)), ("cdft", (2, 1024))]


@pytest.mark.parametrize("kind,n", TILES)
@pytest.mark.parametrize("sweeps", [1, 2, 3, 6])
def test_coarsest_tile_sweeps_equal_float32_sweeps(kind, n, sweeps):
    rng = np.random.default_rng(8)
    shape = tuple(reversed(n))
    rho = (0.8 if kind == "pfc" else 0.3) + 0.03 * rng.uniform(-1, 1, shape)
    vel = [0.05 * rng.standard_normal(shape) for _ in n]
    opts = dict(w_damp=0.5, ncoarse=sweeps, coarsest=4096, tol=1e-300, max_cycles=1, precision=fm.FM_MIXED)
    opts.update(dict(alpha=0.6) if kind == "pfc" else dict(nu=2.362, delta=1e-10))
    res = []
    for coarse in (fm.FM_FP64, fm.FM_MIXED):
        sol = fm.Solver(kind, n, 0.9 if kind == "pfc" else 0.25, coarse_precision=coarse, **opts)
        assert fm.fm_levels(sol.handle) == 1
        sol.set_fields(rho, vel)
        code, info = fm.fm_step_raw(sol.handle, 0.02)
        assert code == fm.FM_ENOCONV and info.cycles == 1
        res.append(info.res)
        sol.close()
    assert abs(res[0] - res[1]) <= 1e-4 * res[1], res
