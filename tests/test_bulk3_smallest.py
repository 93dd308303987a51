"""The smallest grids of the 3D bulk kernel against the oracle: four cells and
two or three velocities an axis."""
import numpy as np
import pytest

import oracle
from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [dvm.FP64, dvm.FP32])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("nv", [(2, 2, 2), (3, 2, 2), (1, 2, 3)])
def test_smallest(nv, scheme, prec):
    cfg = W.base3d(4, nv[0], 1.0, nvy=nv[1], nvz=nv[2], scheme=scheme, Kn=0.3, Lref=1.0, cfl=0.45, bc=[2, 2, 0, 0, 2, 2],
                   init=None)
    # velocities on both sides of zero; with one in x the window puts it at -1
    top = [3.0 if n == 2 else 1.0 for n in nv]
    cfg.update(vxmax=top[0], vymax=top[1], vzmax=top[2])
    F0 = np.random.default_rng(3).uniform(0.5, 1.5, 64 * nv[0] * nv[1] * nv[2]) / np.prod([t + 1 for t in top])   # density near 1
    Fo = F0.copy()
    assert oracle.run(cfg, Fo, 3)["status"] == 0
    s = dvm.Solver(cfg, prec)
    s.set_state(F0)
    s.step(3)
    Fg = s.get_state().astype(np.float64)
    s.close()
    # FP32: three steps, each a handful of roundings of values up to the
    # largest one, and the initial rounding
    tol = 1e-12 if prec == dvm.FP64 else 3e-6
    assert np.abs(Fg - Fo).max() <= tol * np.abs(Fo).max()
