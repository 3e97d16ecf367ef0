"""FP32 on a moving bed: the roundings of its stage kernels decide, through the bed's
coarse grid, whole runs, so they are held bit for bit to recorded runs; and the form
of the kernels follows the bed, which comes to rest and starts again."""
import os

import numpy as np
import pytest

from paper_2002_04889_gb300 import inputs as I
from paper_2002_04889_gb300 import volna

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "moving_bed_fp32_runs.txt")
RUNS = [("hilbert", "open", 12, 60), ("morton", "wall", 9, 41), ("rcm", "absorbing", 21, 30)]


def rupture(n):
    m = I.coast_mesh(n_theta=n, n_xi=2 * n, seed=n)
    return m, I.lake_at_rest_state(m, 0.0), (*I.coast_rupture(m, amplitude=3.0, angle_deg=40.0), 8.0)


def open_context(m, renumber, boundary):
    sv = volna.Solver(32)
    sv.set_params(h_threshold=1e-3, cfl=0.9)
    sv.upload_mesh(m, renumber=renumber)
    if boundary != "wall":
        sv.set_boundary(I.boundary_edges(m, lambda p: np.hypot(p[:, 0], p[:, 1]) > 0.99 * np.hypot(*m.xy.T).max() - 1e3),
                        boundary)
    return sv


def moving_run(renumber, boundary, n, steps):
    m, s, motion = rupture(n)
    with open_context(m, renumber, boundary) as sv:
        sv.set_bed_motion(*motion)
        sv.set_state(s.H, s.Hu, s.Hv, 0.0)
        sv.step(steps)
        return sv.get_state()


def sample(state):
    """Every 11th cell of the three fields, and the time, as exact text."""
    return " ".join(float(v).hex() for a in state[:3] for v in a[::11]) + " " + float(state[3]).hex()


@pytest.mark.parametrize("run", range(len(RUNS)))
def test_recorded_runs(run):
    with open(GOLDEN) as fh:
        ref = [line.split() for line in fh if not line.startswith("#")][run]
    got = sample(moving_run(*RUNS[run])).split()
    assert np.array([float.fromhex(v) for v in ref])[:-1].any()
    assert got == ref


@pytest.mark.parametrize("n", [9, 60])
@pytest.mark.parametrize("boundary", ["wall", "open"])
def test_form_follows_the_bed(n, boundary):
    """One context over a bed at rest, moving, at rest again (a state later than its last
    onset and rise), moving, in other blocks and back, and without motion: each run bit for bit
    that of a fresh context; at rest, that of the uplifted static bed."""
    m, s, motion = rupture(n)
    up, on, rise = motion
    late = float(on.max()) + 2 * rise

    def run(sv, t, H=s.H):
        sv.set_state(H, s.Hu, s.Hv, t)
        sv.step(9)
        return sv.get_state()

    def fresh(t, motion):
        with open_context(m, "hilbert", boundary) as sv:
            if motion:
                sv.set_bed_motion(*motion)
            return run(sv, t)

    static, moving, resting = fresh(0.0, None), fresh(0.0, motion), fresh(late, motion)
    mu = I.Mesh(m.xy, m.tri, m.depth - up, name="uplifted", meta=m.meta)
    with open_context(mu, "hilbert", boundary) as sv:
        lifted = run(sv, late)
    with open_context(m, "hilbert", boundary) as sv:
        got = [run(sv, 0.0)]
        sv.set_bed_motion(*motion)
        got += [run(sv, 0.0), run(sv, late), run(sv, 0.0)]
        sv.set_params(block_cells=128)
        sv.set_params(block_cells=0)
        got += [run(sv, 0.0)]
        sv.set_bed_motion(None)
        got += [run(sv, 0.0)]
    for a, ref in zip(got, (static, moving, resting, moving, moving, static)):
        for x, y in zip(a, ref):
            np.testing.assert_array_equal(x, y)
    for x, y in zip(resting, lifted):
        np.testing.assert_array_equal(x, y)
