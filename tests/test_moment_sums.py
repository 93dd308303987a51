"""Density and temperature of a state from the moment kernels: rows of cells
that end inside a warp, velocity rows that are cut by the ends of a warp's
share, groups that straddle rows, fewer groups than warps."""
import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W

CASES = [
    (2, (32, 4), (2, 1)), (2, (33, 5), (13, 7)), (2, (45, 6), (9, 11)), (2, (64, 4), (33, 3)), (2, (5, 7), (64, 5)),
    (3, (4, 4, 4), (2, 1, 1)), (3, (45, 5, 4), (14, 5, 3)), (3, (33, 4, 7), (7, 6, 5)), (3, (9, 11, 6), (17, 4, 4)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [dvm.FP32, dvm.FP64])
@pytest.mark.parametrize("dim,n,nv", CASES)
def test_moment_sums(dim, n, nv, prec):
    cfg = W.base2d(n[0], n[1], nv[0], 6.0) if dim == 2 else W.base3d(n[0], nv[0], 5.0)
    cfg.update(nx=n[0], ny=n[1], nvx=nv[0], nvy=nv[1])
    if dim == 3:
        cfg.update(nz=n[2], nvz=nv[2])
    s = dvm.Solver(cfg, prec)
    F = np.random.default_rng(11).uniform(0.5, 1.5, s.state_size).astype(s.dtype)
    s.set_state(F)
    m, f = s.moments(), F.astype(np.float64).reshape(s.ncell, s.ncomp, s.nv)
    step = [(cfg[f"v{k}max"] - cfg[f"v{k}min"]) / cfg[f"nv{k}"] for k in ("x", "y", "z")[:dim]]
    v = [cfg[f"v{k}min"] + np.arange(cfg[f"nv{k}"]) * h for k, h in zip(("x", "y", "z"), step)]
    grid = [g.ravel() for g in np.meshgrid(*v[::-1], indexing="ij")[::-1]]
    sums = f[:, 0].sum(1)
    u2 = sum((f[:, 0] @ g / sums) ** 2 for g in grid)
    e2 = (f[:, 0] @ sum(g * g for g in grid) + (2 * f[:, 1].sum(1) if dim == 2 else 0)) / sums
    # the reduced 2D pair stands for a gas with three degrees of freedom;
    # products and velocities rounded a few times each in the state precision
    eps = np.finfo(s.dtype).eps
    assert (np.abs(m["rho"] - sums * np.prod(step)) <= 8 * eps * sums * np.prod(step)).all()
    assert (np.abs(m["T"] - (e2 - u2) / 3) <= 16 * eps * (e2 + 2 * u2)).all()
    s.close()
