"""Device arrays that end before the state does are refused before any kernel
reads or writes them; arrays that end with their allocation, or lie inside a
larger one, are used."""
import threading

import numpy as np
import pytest

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def solver():
    s = dvm.Solver(W.cylinder_adjoint(nx=128, nv=32, nseg=8, steps=1), dvm.FP32)    # 134 MB
    s.init_maxwellian()
    yield s
    s.close()


def _short(s):
    import torch
    one = torch.ones(1, device="cuda")      # in an allocation of 2 MB
    return one.expand(s.state_size)


def test_short_arrays_are_refused(solver):
    s = solver
    F = s.get_state()
    for call in (s.set_state, s.get_state, lambda t: s.adjoint(1, 1, seed=t), s.step_vjp):
        with pytest.raises(dvm.DVMError) as err:
            call(_short(s))
        assert err.value.code == 1
    assert np.array_equal(s.get_state(), F)


@pytest.mark.parametrize("before,after", [(0, 0), (8, 0), (0, 8), (3, 5)])
def test_whole_arrays(solver, before, after):
    import torch
    s = solver
    n = s.state_size
    F = s.get_state()
    t = torch.empty(before + n + after, device="cuda")
    out = t[before:before + n]
    assert np.array_equal(s.get_state(out).cpu().numpy(), F)
    # from a thread that has made no CUDA call yet
    out *= 2
    torch.cuda.synchronize()
    th = threading.Thread(target=s.set_state, args=(out,))
    th.start()
    th.join()
    assert np.array_equal(s.get_state(), 2 * F)
