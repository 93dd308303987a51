"""The fusion of merged control volumes in FP64 where it has an exact answer:
members that all hold the same power of two keep it, since the weighted sum is
that power times the sum of the weights, and their quotient is the power."""
import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W


@pytest.mark.gpu
def test_equal_members_keep_their_value():
    # a step too short to change a value: what is left of it is the fusion
    cfg = W.cylinder_mach2(nx=96, nv=8)
    cfg.update(dt=1e-60, bc=[0] * 6, bc_state=[None] * 6)
    s = dvm.Solver(cfg, dvm.FP64)
    f = 2.0 ** np.random.default_rng(2).integers(-6, 3, 2 * 64)
    s.set_state(np.tile(f, s.ncell))
    F0 = s.get_state()                # the solid cells are 0
    s.step(1)
    F = s.get_state()
    s.close()
    assert (F0 > 0).any() and np.array_equal(F, F0)
