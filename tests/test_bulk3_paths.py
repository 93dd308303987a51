"""The branches of the 3D bulk kernel against the oracle: velocity counts that
put the sign change of v_x on a unit boundary, inside a unit and inside a
group, restarts of the FP64 recurrence (8 and 16 velocities), splits that
start inside a row of groups, and tiles at the edges of 32 x 16 x 4 cells with
the limiter on every face or masked near a sphere."""
import numpy as np
import pytest

import oracle
from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W
from test_parity_3d import bump_init

pytestmark = pytest.mark.gpu

# cells (x, y, z), velocities (x, y, z), window of v_x
CASES = [
    ((33, 17, 5), (13, 3, 3), (-5.0, 5.0)),       # sign change inside a unit
    ((32, 16, 8), (14, 2, 4), (-5.0, 5.0)),       # zero at an odd index
    ((31, 15, 9), (20, 3, 2), (-5.0, 5.0)),       # inside a group, between units
    ((40, 6, 4), (9, 5, 4), (-3.0, 6.0)),         # asymmetric window
    ((6, 20, 7), (33, 2, 3), (-6.0, 6.0)),        # recurrence of 16
    ((5, 5, 6), (64, 2, 2), (-6.0, 6.0)),
    ((4, 4, 4), (2, 2, 2), (-4.0, 4.0)),
]


@pytest.mark.parametrize("prec", [dvm.FP64, dvm.FP32])
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("n,nv,win", CASES)
def test_bulk3_paths(n, nv, win, body, scheme, prec):
    if body and min(n) < 5:
        pytest.skip("no room for an obstacle")
    cfg = W.base3d(n[0], nv[0], 5.0, ny=n[1], nz=n[2], nvy=nv[1], nvz=nv[2], vxmin=win[0], vxmax=win[1],
                   scheme=scheme, Kn=0.3, Lref=1.0, cfl=0.45, bc=[2, 2, 0, 0, 2, 2], init=None)
    if body:
        # the largest sphere that leaves gas cells on every side
        h = max(1.0 / m for m in n)
        cfg.update(shape=3, ra=min(0.3, 0.5 - 1.6 * h), cx=0.503, cy=0.497, cz=0.501)
    cfg["init"] = bump_init(cfg)
    F0 = oracle.initial_state(cfg)
    Fo = F0.copy()
    h = oracle.run(cfg, Fo, 3)
    if h["status"] != 0:
        pytest.skip("not a problem of the method (geometry or moments)")
    s = dvm.Solver(cfg, prec)
    s.set_state(F0)
    s.step(3)
    Fg = s.get_state().astype(np.float64)
    s.close()
    # FP32: three steps, each a handful of roundings of values up to the
    # largest one, and the initial rounding
    tol = 1e-12 if prec == dvm.FP64 else 3e-6
    assert np.abs(Fg - Fo).max() <= tol * np.abs(Fo).max()
