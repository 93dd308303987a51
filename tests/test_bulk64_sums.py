"""The moment sums that an FP64 step leaves with its state, as the checkpoint
holds them: plain sums of at most 16 velocities that join the total, however
many velocities a split has."""
import struct

import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [2, 3])
def test_sums_of_many_velocities(tmp_path, dim):
    # 3D: as many cells as one velocity split fills the chip with: whole rows
    cfg = W.base2d(32, 8, 64, 4.0) if dim == 2 else W.base3d(64, 64, 4.0, ny=64, nz=76, nvy=2, nvz=1)
    cfg.update(scheme=0, bc=[0] * 6, dt=1e-60, Kn=1.0, Lref=1.0, init=None)
    u, rows = 2.0 ** -53, 64 if dim == 2 else 2
    f = np.full((rows, 64), 0.99 * u)    # each lost beside a sum of 1 and above
    f[:, 0] = 1.0
    if dim == 3:
        f[1] = f[1, ::-1]                # a temperature
    s = dvm.Solver(cfg, dvm.FP64)
    nc, ncomp = s.ncell, s.ncomp
    one = np.concatenate([f.ravel(), np.zeros(f.size)]) if dim == 2 else f.ravel()
    s.set_state(np.ascontiguousarray(np.broadcast_to(one, (nc, one.size))).ravel())
    s.step(1)
    path = str(tmp_path / "c.dvm")
    s.save(path)
    s.close()
    raw = open(path, "rb").read()
    nstate, npart = struct.unpack_from("<QQ", raw, 96)
    F = np.frombuffer(raw, np.float64, nstate // 8, 128).reshape(nc, ncomp, -1)[:, 0]
    assert np.array_equal(F, np.broadcast_to(f.ravel(), F.shape))      # the step left the state as it was
    part = np.frombuffer(raw, np.float64, npart // 8, 128 + nstate).reshape(-1, dim + 2, nc)
    got = part[:, 0].astype(np.longdouble).sum(0)
    # a row: 15 additions beside the large value, and the four short sums join
    # the total with a rounding of up to 2 u each
    assert np.abs(got - (rows + f[f < 0.5].astype(np.longdouble).sum())).max() <= (15 + 4 * 2 + 1) * u * rows
