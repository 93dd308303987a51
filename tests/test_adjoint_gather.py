"""The packed FP32 gather of the adjoint against the FP64 one: velocity counts
whose last group is padded, groups that straddle rows and hold both signs of
v_x, fewer groups than the kernel's splits, tiles at the edge of the grid."""
import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("nx,nv", [(40, (13, 7)), (33, (9, 11)), (32, (12, 12)), (48, (6, 5)), (31, (33, 3))])
def test_adjoint_gather(nx, nv, scheme):
    cfg = W.cylinder_adjoint(nx=nx, nv=nv[0], nseg=8, steps=1)
    cfg.update(nvx=nv[0], nvy=nv[1], scheme=scheme)
    rng = np.random.default_rng(3)
    lam = []
    for prec in (dvm.FP32, dvm.FP64):
        s = dvm.Solver(cfg, prec)
        if prec == dvm.FP32:
            s.init_maxwellian()
            # no two differences of neighbours tie, so that both precisions
            # take the same limiter branches
            F = (s.get_state() * rng.uniform(0.9, 1.1, s.state_size)).astype(np.float32)
            seed = rng.uniform(-0.5, 0.5, s.state_size).astype(np.float32)
        s.set_state(F.astype(s.dtype))
        lam.append(np.asarray(s.adjoint(1, 1, seed=seed.astype(s.dtype))["lambda0"], dtype=np.float64))
        s.close()
    # one transposed step: some twenty products a value, rounded once each,
    # and moment sums of the velocities
    assert np.abs(lam[0] - lam[1]).max() <= 1e-5 * np.abs(lam[1]).max()
