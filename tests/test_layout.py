"""Conversion between the public state layout and the device layout: sizes on
both sides of the 32-cell by 512-byte tiles, padded and unpadded velocity
rows, arrays that start on a 16-byte vector and ones that do not."""
import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W

CASES = [
    # dim, cells, velocities: one tile, ragged tiles, padded rows (velocity
    # counts that are no multiple of the vector), several tiles of velocities
    (2, (4, 4), (1, 1)), (2, (32, 5), (16, 8)), (2, (33, 7), (13, 3)), (2, (71, 9), (17, 17)), (2, (40, 6), (64, 6)),
    (3, (4, 4, 4), (1, 1, 1)), (3, (32, 4, 5), (8, 4, 2)), (3, (35, 5, 6), (7, 3, 5)), (3, (65, 4, 4), (18, 3, 4)),
]


def _cfg(dim, n, nv):
    cfg = W.base2d(n[0], n[1], nv[0], 6.0) if dim == 2 else W.base3d(n[0], nv[0], 5.0)
    cfg.update(nx=n[0], ny=n[1], nvx=nv[0], nvy=nv[1])
    if dim == 3:
        cfg.update(nz=n[2], nvz=nv[2])
    return cfg


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [dvm.FP32, dvm.FP64])
@pytest.mark.parametrize("dim,n,nv", CASES)
def test_layout_round_trip(dim, n, nv, prec):
    import torch
    cfg = _cfg(dim, n, nv)
    s = dvm.Solver(cfg, prec)
    F = np.random.default_rng(5).uniform(0.5, 1.5, s.state_size).astype(s.dtype)
    size = s.state_size
    for off in (0, 1):                       # on a vector, and one element past it
        d = torch.zeros(size + 2, dtype=torch.float32 if prec == dvm.FP32 else torch.float64, device="cuda")
        d[off:off + size] = torch.as_tensor(F, device="cuda")
        torch.cuda.synchronize()
        s.set_state(d[off:off + size])
        assert np.array_equal(s.get_state(), F)
        s.set_state(2 * F)
        out = torch.full((size + 2,), -1.0, dtype=d.dtype, device="cuda")
        torch.cuda.synchronize()
        s.get_state(out[off:off + size])
        assert np.array_equal(out[off:off + size].cpu().numpy(), 2 * F)
        assert bool((out[:off] == -1).all()) and bool((out[off + size:] == -1).all())
        # every velocity sits where the kernels look for it: the density and
        # the momentum of the device layout against sums of the public one
        m, f = s.moments(), (2 * F).astype(np.float64).reshape(s.ncell, s.ncomp, s.nv)[:, 0]
        v = [cfg[f"v{k}min"] + np.arange(cfg[f"nv{k}"]) * ((cfg[f"v{k}max"] - cfg[f"v{k}min"]) / cfg[f"nv{k}"])
             for k in ("x", "y", "z")[:dim]]
        grid = np.meshgrid(*v[::-1], indexing="ij")[::-1]
        # each sum: at most nv products, rounded once each in the state
        # precision, and the table's velocities rounded once
        eps = np.finfo(s.dtype).eps
        for k, g in zip(("ux", "uy", "uz"), grid):
            g = g.ravel()
            ref = f @ g / f.sum(1)
            tol = 8 * eps * (f @ np.abs(g)) / f.sum(1) + 1e-300
            assert (np.abs(m[k] - ref) <= tol).all(), k
    s.close()
