"""A checkpoint whose moment sums are grouped in another number of velocity
splits than the loading context uses: the slots are summands of each cell's
moments, so the run continues as from the same sums."""
import struct

import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W

pytestmark = pytest.mark.gpu

S_AT, PART_AT, HEADER = 28, 104, 128


def _regroup(raw, split):
    """The file with every slot's sums moved into `split` times as many slots
    (or, split = 0, all added into one slot)."""
    S, = struct.unpack_from("<i", raw, S_AT)
    nstate, npart = struct.unpack_from("<QQ", raw, PART_AT - 8)
    part = np.frombuffer(raw, np.float64, npart // 8, HEADER + nstate).reshape(S, -1)
    if split:
        new = np.zeros((S * split, part.shape[1]))
        new[::split] = part
    else:
        new = part.sum(0, keepdims=True)
    head = bytearray(raw[:HEADER])
    struct.pack_into("<i", head, S_AT, len(new))
    struct.pack_into("<Q", head, PART_AT, new.nbytes)
    return bytes(head) + raw[HEADER:HEADER + nstate] + new.tobytes() + raw[HEADER + nstate + npart:]


@pytest.mark.parametrize("split", [0, 2, 30])
@pytest.mark.parametrize("cfg", [W.cylinder_mach2(nx=48, nv=16), W.sphere_mach15(n=24, nv=8)], ids=["2d", "3d"])
def test_load_other_split_count(tmp_path, cfg, split):
    a, b = str(tmp_path / "a.dvm"), str(tmp_path / "b.dvm")
    s = dvm.Solver(cfg, dvm.FP64)
    s.init_maxwellian()
    s.step(3)
    s.save(a)
    raw = open(a, "rb").read()
    S, = struct.unpack_from("<i", raw, S_AT)
    open(b, "wb").write(_regroup(raw, split))
    s.step(3)
    ref = s.get_state()
    s.close()
    t = dvm.Solver(cfg, dvm.FP64)
    if split and S * split > t.nv // 2:
        with pytest.raises(dvm.DVMError):      # more slots than velocity groups: no checkpoint of this library
            t.load(b)
        t.close()
        return
    t.load(b)
    t.step(3)
    got = t.get_state()
    t.close()
    # the sums differ by their grouping alone
    assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()
