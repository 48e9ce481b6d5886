"""A context's work stays on its own stream, also where a scalar result goes to
device memory: gl_stress and gl_failure_index come back while the default stream
is still busy (a spin of a second or so against calls of well under a
millisecond), with the results of host arrays."""
import ctypes as C

import numpy as np
import pytest

from paper_1707_04228_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_device_peak_does_not_wait_for_the_default_stream(gl_lib, cuda_ok):
    import torch
    from paper_1707_04228_gb300 import lib
    st = torch.cuda.Stream()
    s = lib.Solver.from_laminate(inputs.corner_mini(n_arc=5, n_limb=1, n_width=3, nel_layer=1, angles=(0, 45, 90),
                                                    nsub=(3, 1, 1), nev=4, limb_L=3.0, width=3.0), stream=st)
    u = 1e-3 * inputs.random_vector(s.n_dof, 11)
    ref = (s.stress(u)[2], s.failure_index(u)[1])
    ud = torch.from_numpy(u).cuda()
    out = torch.empty(2, s.n_elem, dtype=torch.float64, device="cuda")
    peak = torch.zeros(2, dtype=torch.float64, device="cuda")
    elem = C.c_int64()
    at = lambda t: C.c_void_p(t.data_ptr())
    calls = [lambda: s.lib.gl_stress(s.ctx, at(ud), at(out[0]), at(out[1]), at(peak)),
             lambda: s.lib.gl_failure_index(s.ctx, at(ud), 61.0, 97.0, at(out[0]), at(peak[1:]), C.byref(elem))]
    for call in calls:
        assert call() == 0
    peak.zero_()
    for call in calls:
        torch.cuda.synchronize()
        busy = torch.cuda.Event()
        torch.cuda._sleep(2_000_000_000)
        busy.record()
        rc = call()
        still = not busy.query()
        torch.cuda.synchronize()
        assert rc == 0 and still
    assert tuple(peak.tolist()) == ref
    s.close()
