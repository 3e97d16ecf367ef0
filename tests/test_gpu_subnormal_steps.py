"""FP64 literal steps at the bottom of the number range equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2002_04889_gb300 import inputs as I
from paper_2002_04889_gb300 import volna

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unfused", [0, 1])
@pytest.mark.parametrize("top", [3, 1000, 2 ** 54, 2 ** 60, 2 ** 117])
def test_subnormal_momenta(top, unfused):
    """Films of 1e-160 m whose momenta are up to `top` times the smallest positive double:
    a step halves odd multiples of it."""
    m = I.flat_basin_mesh(12, 1.0, 0.0)
    rng = np.random.default_rng(top % 997)
    H = 1e-160 * (1 + rng.random(m.nc))
    Hu, Hv = np.ldexp(np.floor(rng.random((2, m.nc)) * min(top, 2.0 ** 53)) * 2 + 1, -1074) * max(1, top // 2 ** 53)
    ref = O.OracleMesh.from_mesh(m).run(O.params(h_threshold=0.0, dt_fixed=1.0), (H, Hu, -Hv, 0.0), 3)
    with volna.Solver(64) as sv:
        sv.set_params(h_threshold=0.0, dt_fixed=1.0, rk_unfused=unfused)
        sv.upload_mesh(m)
        sv.set_state(H, Hu, -Hv, 0.0)
        sv.step(3)
        got = sv.get_state()
    assert ref["Hu"].any()
    for a, k in zip(got, ("H", "Hu", "Hv")):
        np.testing.assert_array_equal(a.view(np.int64), ref[k].view(np.int64))
