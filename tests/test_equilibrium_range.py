"""The FP64 equilibrium of the bulk kernels over the width of the v_x grid in
units of sqrt(T), up to grids that hardly resolve the Maxwellian, with its
peak at every place of a row: a step against the oracle, and each value of the
Maxwellian, down to its far tail, against extended precision."""
import math

import numpy as np
import pytest

import oracle
from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FRAC = 0.05         # share of a cell's gas at the next velocity in x


def _grid(cfg, ax):
    n, a, b = cfg[f"nv{ax}"], cfg[f"v{ax}min"], cfg[f"v{ax}max"]
    return a + np.arange(n) * ((b - a) / n)


def _problem(dim, nvx, ratio, place, frac=FRAC, **opt):
    """A problem whose gas has dv_x = ratio sqrt(T) and a window with v_x = 0
    at `place`, and its state: at rest (frac = 0), or the cells' mean v_x
    beside the velocities around that place (a mean speed of many sqrt(T)
    would cancel in T); the width of the rest of the distribution gives T."""
    dv, T = 0.5, (0.5 / ratio) ** 2
    rest = 3 * T - frac * (1 - frac) * dv * dv
    assert rest > 0
    lo = -place * dv
    if dim == 2:
        cfg = W.base2d(12, 9, nvx, 1.0, nvy=3, **opt)
        cfg.update(vymin=-1.0, vymax=2.0)
    else:
        # v_y and v_z at +-a
        cfg = W.base3d(9, nvx, 1.0, ny=6, nz=5, nvy=2, nvz=2, **opt)
        a = math.sqrt(0.5 * rest)
        cfg.update(vymin=-a, vymax=3 * a, vzmin=-a, vzmax=3 * a)
    cfg.update(vxmin=lo, vxmax=lo + nvx * dv, bc=[0] * 6, init=None, Lref=1.0)
    _relaxing(cfg, dim)
    nc, rng = cfg["nx"] * cfg["ny"] * cfg["nz"], np.random.default_rng(7)
    c = np.arange(nc)
    rho = rng.uniform(0.8, 1.2, nc) if frac else np.ones(nc)
    k = np.clip(place + c % 7 - 3, 0, nvx - 2) if frac else np.full(nc, place)
    if dim == 2:
        F = np.zeros((nc, 2, 3, nvx))
        F[c, 0, 1, k] = rho * (1 - frac)
        if frac:
            F[c, 0, 1, k + 1] = rho * frac
        F[:, 1] = F[:, 0] * (0.5 * rest)
    else:
        F = np.zeros((nc, 2, 2, nvx))
        F[c, :, :, k] = (rho * (1 - frac) / 4)[:, None, None]
        if frac:
            F[c, :, :, k + 1] = (rho * frac / 4)[:, None, None]
    F /= np.prod([_grid(cfg, k)[1] - _grid(cfg, k)[0] for k in ("x", "y", "z")[:dim]])
    return cfg, F.ravel()


def _relaxing(cfg, dim):
    """The time step of Courant number 0.4, and dt/tau = 0.3 at density 1."""
    cfg["dt"] = 0.4 / sum(np.abs(_grid(cfg, k)).max() * cfg["n" + k] for k in ("x", "y", "z")[:dim])
    cfg["Kn"] = cfg["dt"] / 0.3 * math.sqrt(2.0) / (math.sqrt(math.pi) / 2.0)


def _step_both(cfg, F0):
    Fo = F0.copy()
    assert oracle.run(cfg, Fo, 1)["status"] == 0
    s = dvm.Solver(cfg, dvm.FP64)
    s.set_state(F0)
    s.step(1)
    Fg = s.get_state()
    s.close()
    assert np.abs(Fg - Fo).max() <= 1e-12 * np.abs(Fo).max()


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("opt", ["", "imex", "shakhov"])
@pytest.mark.parametrize("ratio", [0.5, 1.0, 1.5, 2.4, 2.6, 4.0, 6.0])
@pytest.mark.parametrize("nvx", [12, 20, 32, 33, 40, 64])
@pytest.mark.parametrize("dim", [2, 3])
def test_step_against_oracle(dim, nvx, ratio, opt, scheme):
    for place in range(3, nvx - 1, 7):
        cfg, F0 = _problem(dim, nvx, ratio, place, scheme=scheme, time_scheme=int(opt == "imex"),
                           model=int(opt == "shakhov"), Pr=2.0 / 3.0)
        _step_both(cfg, F0)


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("ratio", [1.5, 2.4, 2.6, 3.0])
@pytest.mark.parametrize("nvx,places", [(12, (5,)), (20, (11, 14)), (33, (14, 23)), (40, (18, 30)), (64, (5, 31, 45, 60))])
@pytest.mark.parametrize("dim", [2, 3])
def test_conservative_step_against_oracle(dim, nvx, places, ratio, scheme):
    """Maxwellians about the velocity `place` of the window, which exist on
    grids this coarse with parameters other than the direct moments."""
    dv, T = 0.5, (0.5 / ratio) ** 2
    c = math.sqrt(T)
    for place in places:
        cfg = W.base2d(12, 9, nvx, 1.0, nvy=10) if dim == 2 else W.base3d(9, nvx, 1.0, ny=6, nz=5, nvy=8, nvz=8)
        nc, rng = cfg["nx"] * cfg["ny"] * cfg["nz"], np.random.default_rng(7)
        w = 5 * c if dim == 2 else 4 * c
        cfg.update(vxmin=-place * dv, vxmax=(nvx - place) * dv, vymin=-w, vymax=w, vzmin=-w, vzmax=w, bc=[0] * 6, Lref=1.0,
                   scheme=scheme, conservative=1,
                   init=dict(rho=rng.uniform(0.8, 1.2, nc), ux=rng.uniform(-0.4, 0.4, nc) * dv,
                             uy=rng.uniform(-0.1, 0.1, nc) * c, uz=0.0, T=T))
        _relaxing(cfg, dim)
        F0 = oracle.initial_state(cfg)
        _step_both(cfg, F0)


@pytest.mark.parametrize("ratio", [0.5, 1.0, 1.5, 2.4, 4.0])
@pytest.mark.parametrize("nvx,places", [(20, (0, 3, 7, 8, 19)), (33, (1, 15, 16, 31)), (64, (0, 15, 30, 47, 63))])
@pytest.mark.parametrize("dim", [2, 3])
def test_each_value(dim, nvx, places, ratio):
    """A uniform gas at rest with all its f at v_x = 0: after a step every
    other value of f is r M alone."""
    for place in places:
        cfg, F0 = _problem(dim, nvx, ratio, place, frac=0.0, scheme=1)
        s = dvm.Solver(cfg, dvm.FP64)
        s.set_state(F0)
        s.step(1)
        F = s.get_state().reshape(s.ncell, s.ncomp, -1)[:, 0].reshape(s.ncell, -1, nvx)
        r = np.longdouble(s.dt) / np.longdouble(s.tau0)
        s.close()
        v = [_grid(cfg, k).astype(np.longdouble) for k in ("x", "y", "z")[:dim]]
        f = F0.reshape(len(F), 2 if dim == 2 else 1, -1)[0].astype(np.longdouble)
        d2 = sum(g * g for g in np.meshgrid(*v[::-1], indexing="ij"))
        rho = f[0].sum() * np.prod([g[1] - g[0] for g in v])
        T = ((f[0] * d2.ravel()).sum() + (2 * f[1].sum() if dim == 2 else 0)) / f[0].sum() / 3
        x = d2 / (2 * T)
        pi = np.longdouble("3.14159265358979323846")
        M = (r * rho * rho * (1 / (2 * pi * T)) ** (np.longdouble(dim) / 2) * np.exp(-x)).reshape(-1, nvx)
        x = x.reshape(M.shape)
        away = np.arange(nvx) != place
        M, x, F = M[:, away], x[:, away], F[:, :, away]
        far = M < 1e-290           # towards the smallest numbers
        assert (F[:, far] <= 1e-289).all() and (F >= 0).all()
        # The exponent carries the rounding of T (four operations), of the
        # scale (three) and of its product, the factors some twenty
        u = np.longdouble(2.0) ** -53
        assert (np.abs(F[:, ~far] - M[~far]) <= ((8 * x + 24) * u * M)[~far]).all()
