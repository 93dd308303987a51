"""The moment sums that a 3D FP32 step leaves with its state, as the
checkpoint holds them: plain FP32 sums of at most 32 velocities before the
compensated one, whatever the length of a v_x row."""
import struct

import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W


@pytest.mark.gpu
def test_sums_of_a_long_row(tmp_path):
    # as many cells as one velocity split fills the chip with: whole rows
    cfg = W.base3d(64, 64, 4.0, ny=64, nz=76, nvy=2, nvz=1, scheme=0, bc=[0] * 6, dt=1e-20, Kn=1.0, Lref=1.0, init=None)
    u = 2.0 ** -24
    f = np.full((2, 64), 0.99 * u)       # each lost beside a sum of 1 and above
    f[0, 0] = f[1, 63] = 1.0
    s = dvm.Solver(cfg, dvm.FP32)
    nc = s.ncell
    s.set_state(np.ascontiguousarray(np.broadcast_to(f.astype(np.float32).ravel(), (nc, 128))).ravel())
    s.step(1)
    path = str(tmp_path / "c.dvm")
    s.save(path)
    s.close()
    raw = open(path, "rb").read()
    nstate, npart = struct.unpack_from("<QQ", raw, 96)
    F = np.frombuffer(raw, np.float32, nstate // 4, 128).reshape(nc, 128)
    part = np.frombuffer(raw, np.float32, npart // 4, 128 + nstate).reshape(-1, 5, nc)
    want = F.astype(np.float64).sum(1)
    assert np.abs(want - 2).max() < 1e-5           # the step left the state as it was
    got = part.astype(np.float64).sum(0)[0]
    # 31 additions beside a sum of 1, the last large value, the final sum
    assert np.abs(got - want).max() <= 35 * u
