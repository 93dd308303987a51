"""The equilibrium of the first-order FP32 step value by value: a uniform gas
with all its f at one velocity, so that after a step every other value of f is
r M alone (the Shakhov gas has no heat flux).  The gas is fast against its
thermal speed in one case (an exponent formed from large terms would lose its
last digits) and dense and cold in the other (the exponential falls below the
smallest normal number while M does not)."""
import math

import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("place,rho,T", [(63, 1.0, 0.25), (2, 1.0, 0.25), (32, 2.0 ** 17, 2.0 ** -6), (30, 2.0 ** 17, 2.0 ** -4)])
def test_first_order_values(place, rho, T, model):
    dv, nvx = 0.5, 64
    cfg = W.base2d(40, 12, nvx, 1.0, nvy=3, scheme=0, model=model, Pr=2.0 / 3.0, Lref=1.0, init=None)
    cfg.update(vxmin=-16.0, vxmax=16.0, vymin=-1.0, vymax=2.0)
    cfg["dt"] = 0.4 / (16.0 * 40 + 1.0 * 12)
    cfg["Kn"] = cfg["dt"] * rho / 0.25 * math.sqrt(2.0) / (math.sqrt(math.pi) / 2.0)
    nc = 40 * 12
    F0 = np.zeros((nc, 2, 3, nvx), np.float32)
    F0[:, 0, 1, place] = rho / dv            # powers of two: the moments are exact
    F0[:, 1, 1, place] = rho / dv * (1.5 * T)
    s = dvm.Solver(cfg, dvm.FP32)
    s.set_state(F0.ravel())
    s.step(1)
    F = s.get_state().reshape(F0.shape)[:, 0].astype(np.float64)
    r = s.dt / s.tau0 * rho
    s.close()
    vx = -16.0 + dv * np.arange(nvx)
    x = ((vx - vx[place]) ** 2 + (np.arange(3) - 1.0)[:, None] ** 2) / (2 * T)
    A = r * rho / (2 * math.pi * T)
    M = A * np.exp(-x)
    away = np.ones((3, nvx), bool)
    away[1, place] = False
    # rounding of the exponent (T and the scale seven, the difference two) and
    # of the factors, the exponential's own error, the spacing of the smallest
    # numbers
    tol = (10 * x + 32) * 2.0 ** -24 * M + A * 2.0 ** -148
    assert (np.abs(F - M) <= tol)[:, away].all()
