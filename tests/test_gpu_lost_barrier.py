"""Steps in one launch whose thread blocks lose one another: every wait ends after its
limit, the call reports VG_ETIMEOUT, and nothing is left behind for later steps."""
import ctypes

import numpy as np
import pytest

from paper_2002_04889_gb300 import inputs as I
from paper_2002_04889_gb300 import volna

pytestmark = pytest.mark.gpu


def lose_arrival(sv, polls):
    f = volna.load().vg_debug_lose_arrival
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_uint32], ctypes.c_int
    assert f(sv.ctx, polls) == volna.VG_OK


def context(m, s):
    sv = volna.Solver(32)
    sv.set_params(h_threshold=1e-5, cfl=0.9)
    sv.upload_mesh(m)
    sv.set_gauges(np.array([[0.0, 0.0], [0.2, 0.1]]))
    sv.set_state(s.H, s.Hu, s.Hv, 0.0)
    return sv


@pytest.mark.parametrize("polls", [1, 300])
@pytest.mark.parametrize("n", [1, 9, 66, 300])
def test_steps_give_up(n, polls):
    m = I.thacker_mesh(n=n)
    s = I.thacker_initial_state(m)
    with context(m, s) as sv:
        sv.step(7)
        ref = [*sv.get_state(), *sv.gauges()]
    with context(m, s) as sv:
        sv.step(2)
        lose_arrival(sv, polls)
        for _ in range(2):                       # the state is lost until another is set
            with pytest.raises(volna.VolnaError) as e:
                sv.step(5)
            assert e.value.code == volna.VG_ETIMEOUT
        sv.set_state(s.H, s.Hu, s.Hv, 0.0)
        sv.step(3)
        sv.step(4)
        for a, b in zip([*sv.get_state(), *sv.gauges()], ref):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("polls", [1, 300])
@pytest.mark.parametrize("n", [1, 9, 66, 300])
def test_a_callers_step_gives_up(n, polls):
    import torch
    m = I.thacker_mesh(n=n)
    s = I.thacker_initial_state(m)
    with context(m, s) as sv:
        perm = torch.from_numpy(sv.permutation().astype(np.int64)).cuda()
        w = torch.empty(3, m.nc, device="cuda")
        w[:, perm] = torch.from_numpy(np.stack([s.H - m.vertex_mean(m.depth), s.Hu, s.Hv])).float().cuda()
        out, again = torch.empty_like(w), torch.empty_like(w)
        sv.step(2)
        dt = volna.vg_step_noalloc(sv.ctx, w.data_ptr(), out.data_ptr(), 0.0)
        sv.step(3)
        ref = [*sv.get_state(), *sv.gauges()]
        sv.set_state(s.H, s.Hu, s.Hv, 0.0)
        sv.step(2)
        lose_arrival(sv, polls)
        with pytest.raises(volna.VolnaError) as e:
            volna.vg_step_noalloc(sv.ctx, w.data_ptr(), again.data_ptr(), 0.0)
        assert e.value.code == volna.VG_ETIMEOUT
        sv.step(3)                               # the context's own run has noticed nothing
        for a, b in zip([*sv.get_state(), *sv.gauges()], ref):
            np.testing.assert_array_equal(a, b)
        assert volna.vg_step_noalloc(sv.ctx, w.data_ptr(), again.data_ptr(), 0.0) == dt
        assert torch.equal(out, again)
