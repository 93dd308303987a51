"""The branches of the FP64 2D bulk kernel against the oracle: odd velocity
counts (groups that straddle rows, one of them with both signs of v_y),
restarts of the Maxwellian's recurrence (8 and 16 velocities), splits that
start inside a row, ragged tiles of 32 x 8 cells, periodic and zero-gradient
sides, with the limiter on every face or masked near an obstacle."""
import numpy as np
import pytest

import oracle
from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [
    ((33, 9), (13, 7), [0] * 6), ((32, 8), (16, 16), [2, 2, 2, 2, 0, 0]), ((31, 17), (9, 11), [2, 2, 0, 0, 0, 0]),
    ((40, 23), (33, 3), [0, 0, 2, 2, 0, 0]), ((5, 6), (64, 2), [0] * 6), ((70, 64), (6, 5), [2, 2, 2, 2, 0, 0]),
]


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("n,nv,bc", CASES)
def test_bulk64_paths(n, nv, bc, body, model, scheme):
    if body and min(n) < 9:
        pytest.skip("no room for an obstacle")
    X, Y = np.meshgrid((np.arange(n[0]) + 0.5) / n[0], (np.arange(n[1]) + 0.5) / n[1])
    init = dict(rho=(1 + 0.2 * np.sin(2 * np.pi * X) * np.cos(2 * np.pi * Y)).ravel(), ux=(0.3 * np.cos(2 * np.pi * Y)).ravel(),
                uy=(0.2 * np.sin(2 * np.pi * (X + Y))).ravel(), uz=0.0, T=(1 + 0.1 * np.cos(2 * np.pi * X)).ravel())
    cfg = W.base2d(n[0], n[1], nv[0], 5.0, nvy=nv[1], scheme=scheme, Kn=0.3, Lref=1.0, cfl=0.45, bc=list(bc), init=init,
                   model=model, Pr=2.0 / 3.0)
    if body:
        h = max(1.0 / m for m in n)
        cfg.update(shape=1, ra=min(0.25, 0.5 - 2.2 * h), cx=0.503, cy=0.497)
    F0 = oracle.initial_state(cfg)
    Fo = F0.copy()
    if oracle.run(cfg, Fo, 3)["status"] != 0:
        pytest.skip("not a problem of the method (geometry or moments)")
    s = dvm.Solver(cfg, dvm.FP64)
    s.set_state(F0)
    s.step(3)
    Fg = s.get_state()
    s.close()
    assert np.abs(Fg - Fo).max() <= 1e-12 * np.abs(Fo).max()
