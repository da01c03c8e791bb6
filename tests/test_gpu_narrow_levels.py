"""Levels narrower than a tile: what sweeps them is chosen by the tiles they take,
not by their points alone, and the sweeps are the same either way."""
import numpy as np
import pytest

from oracle import channel as Ch
from oracle import gradflow as GF
from oracle import scheme as S
from paper_1503_07416_gb300 import fm
from tests.test_gpu_fixed_point import test_source_and_residual_rows as _rows
from tests.test_gpu_fused import _lagged_ghost_update

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1503_07416_gb300 import build
    build.build_library()
    fm.lib()


def _one_cycle(kind, n, coarse, ncoarse):
    """(residual left by one damped cycle, kernels of the step)."""
    rng = np.random.default_rng(9)
    shape = tuple(reversed(n))
    rho = (0.8 if kind == "pfc" else 0.3) + 0.03 * rng.uniform(-1, 1, shape)
    vel = [0.05 * rng.standard_normal(shape) for _ in n]
    kw = dict(alpha=0.6) if kind == "pfc" else dict(nu=2.362, delta=1e-10)
    sol = fm.Solver(kind, n, 0.9 if kind == "pfc" else 0.25, precision=fm.FM_MIXED, coarse_precision=coarse, w_damp=0.5,
                    ncoarse=ncoarse, coarsest=8192, tol=1e-300, max_cycles=1, **kw)
    assert fm.fm_levels(sol.handle) == 1
    sol.set_fields(rho, vel)
    before = fm.fm_profile_read(sol.handle)[2]
    code, info = fm.fm_step_raw(sol.handle, 0.02)
    launches = fm.fm_profile_read(sol.handle)[2] - before
    sol.close()
    assert code == fm.FM_ENOCONV and info.cycles == 1
    return info.res, launches


# (tiles of 8 x 4 points, at most 304 of them on a GB300): narrow levels of fewer
# points than 128 x 64 that take more tiles, and squarer ones that take as many or fewer
@pytest.mark.parametrize("kind,n,tiled", [("pfc", (2, 2048), False), ("pfc", (4, 2000), False), ("cdft", (4096, 2), False),
                                          ("pfc", (110, 90), False), ("pfc", (128, 76), True), ("pfc", (2, 1024), True),
                                          ("cdft", (1024, 8), True), ("pfc", (92, 98), True)])
def test_coarsest_level_route(kind, n, tiled):
    """Two launches of two sweeps on tiles; or two conversions and eight colour
    launches.  The residual after the cycle against the float32 solve, a separate
    implementation: they differ by the float32 rounding of a few dozen updates, a
    few 1e-6 of it; bound 1e-4."""
    res, launches = _one_cycle(kind, n, fm.FM_FP64, 4)
    ref, _ = _one_cycle(kind, n, fm.FM_MIXED, 4)
    assert abs(res - ref) <= 1e-4 * ref
    _, more = _one_cycle(kind, n, fm.FM_FP64, 6)
    assert more - launches == (1 if tiled else 4)


@pytest.mark.parametrize("vel_of", ["ordinary", "spike"])
@pytest.mark.parametrize("n", [(2, 600), (8, 34), (10, 66), (16, 32), (16, 2), (18, 34)])
def test_narrow_channel_rows(n, vel_of):
    """The channel's source and residual on 8 x 32 tiles (up to 16 points wide) and
    just beyond: rows, ghosts and ragged tiles as in test_gpu_fixed_point."""
    _rows("pfc", n, "walls", vel_of)


# a level of its own: narrow ones swept by colour launches and on tiles, the float64
# flow on either side of its line, a level of 2.1 tiles a multiprocessor
SWEEPS = [("gradflow", (2, 8192), fm.FM_MIXED, "colour"), ("gradflow", (8192, 2), fm.FM_MIXED, "tiles"),
          ("gradflow", (2, 4096), fm.FM_FP64, "colour"), ("gradflow", (128, 128), fm.FM_FP64, "tiles"),
          ("gradflow", (256, 160), fm.FM_FP64, "colour"), ("gradflow", (66, 1000), fm.FM_MIXED, "tiles"),
          ("walls", (2, 8192), fm.FM_MIXED, "colour"), ("walls", (8, 1024), fm.FM_MIXED, "tiles"),
          ("walls", (2, 4096), fm.FM_FP64, "colour"), ("walls", (150, 250), fm.FM_FP64, "colour"),
          ("walls", (136, 144), fm.FM_FP64, "tiles"), ("walls", (256, 256), fm.FM_FP64, "tiles")]


@pytest.mark.parametrize("model,n,precision,route", SWEEPS)
def test_fused_solvers_route(model, n, precision, route, monkeypatch):
    """Launches of two more sweeps: four per colour, one of two sweeps on float32
    tiles, two on float64 tiles.  The residual after a cycle of six sweeps against the
    oracle's, with the bounds of test_gpu_fused."""
    rng = np.random.default_rng(5)
    shape, h, s = tuple(reversed(n)), 0.9, 0.02
    rho = 0.8 + 0.05 * rng.uniform(-1, 1, shape)
    P = S.Params(kind=S.PFC, dim=2, h=h, s=s, alpha=0.6, w_damp=0.5)
    opts = S.SolverOpts(coarsest=8192, ncoarse=6)
    if model == "gradflow":
        kw, vel, W = dict(model=fm.FM_GRADFLOW), None, None
        f, g = GF.source(rho, P), GF.initial_iterate(rho, P)
        GF.vcycle(g, f, P, opts)
        want = S.res_norm(GF.residual(g, f, P), h)
    else:
        monkeypatch.setattr(Ch, "point_update", _lagged_ghost_update)
        W = Ch.Walls(-2e-3, 1e-3)
        kw, vel = dict(walls=fm.FM_WALLS_Y, u_wall=(W.u_bot, W.u_top)), [1e-3 * rng.standard_normal(shape) for _ in n]
        c = Ch.Coeffs(rho, Ch.vorticity(vel, h, W))
        f, g = Ch.source(rho, vel, c.om, P, W), Ch.initial_iterate(rho, vel, P, W)
        Ch.vcycle(g, f, c, P, W, opts)
        want = S.res_norm(Ch.residual(g, f, c, P, W), h)
    count, res = [], 0.0
    for sweeps in (4, 6):
        sol = fm.Solver("pfc", n, h, alpha=0.6, precision=precision, w_damp=0.5, ncoarse=sweeps, coarsest=8192, tol=1e-300,
                        max_cycles=1, **kw)
        assert fm.fm_levels(sol.handle) == 1
        sol.set_fields(rho, vel)
        before = fm.fm_profile_read(sol.handle)[2]
        code, info = fm.fm_step_raw(sol.handle, s)
        count.append(fm.fm_profile_read(sol.handle)[2] - before)
        res = info.res
        sol.close()
        assert code == fm.FM_ENOCONV and info.cycles == 1
    assert count[1] - count[0] == (4 if route == "colour" else (2 if precision == fm.FM_FP64 else 1))
    bound = 1e-3 if model == "walls" else (1e-7 if precision == fm.FM_FP64 else 1e-4)
    assert abs(res - want) <= bound * want, (res, want)
