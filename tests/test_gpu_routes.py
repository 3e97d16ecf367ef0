"""Which route a call takes: launches of many steps, a caller's step in one launch and
kept adjoint recordings run where they should and nowhere else; and contexts that
overlap on the GPU through them."""
import ctypes
import threading

import numpy as np
import pytest

from paper_2002_04889_gb300 import inputs as I
from paper_2002_04889_gb300 import volna

pytestmark = pytest.mark.gpu


def joined(sv):
    """(thread blocks, variant, launches) of the context's launches of many steps."""
    f = volna.load().vg_debug_joined
    g, c, n = ctypes.c_int32(), ctypes.c_int32(), ctypes.c_int64()
    f.argtypes = [ctypes.c_void_p, *map(ctypes.POINTER, (ctypes.c_int32, ctypes.c_int32, ctypes.c_int64))]
    assert f(sv.ctx, ctypes.byref(g), ctypes.byref(c), ctypes.byref(n)) == volna.VG_OK
    return g.value, c.value, n.value


def context(m, precision=32, **prm):
    sv = volna.Solver(precision)
    sv.set_params(h_threshold=1e-5, cfl=0.9, **prm)
    sv.upload_mesh(m)
    s = I.thacker_initial_state(m)
    sv.set_state(s.H, s.Hu, s.Hv, 0.0)
    return sv


# Blocks of 256 cells (from n = 198): four CTAs per SM hold 608 of them on 152 SMs, five
# hold 760; the variant with fewer rounds (four of equals), up to three rounds.
# n = 305: 727 blocks, 460: 1654 (three rounds of both), 539: 2270, 541: 2287
@pytest.mark.parametrize("n,variant", [(1, 4), (66, 4), (110, 4), (223, 4), (305, 5), (460, 4), (539, 5), (541, 0)])
def test_steps_are_joined_up_to_three_rounds(n, variant):
    m = I.thacker_mesh(n=n, half_width=0.02 * n, h0=0.002 * n, alpha=0.02 * n, r0=0.016 * n)
    with context(m) as sv:
        sv.step(5)
        sv.step(4)
        grid, ctas, launches = joined(sv)
        assert (launches, grid > 0) == ((2, True) if variant else (0, False))
        assert not variant or ctas == variant
        sv.profile(True)                         # kernel by kernel
        sv.step(2)
        sv.profile(False)
        sv.set_params(rk_unfused=1)
        sv.step(2)
        sv.set_params(rk_unfused=0)
        assert joined(sv)[2] == launches
        sv.step(2)
        assert joined(sv)[2] == launches + (variant > 0)


def test_what_is_not_joined():
    m = I.thacker_mesh(n=30)
    s = I.thacker_initial_state(m)
    for precision, prm in ((64, {}), (64, dict(fp64_literal=0)), (32, dict(block_cells=192, block_threads=384))):
        with context(m, precision, **prm) as sv:
            sv.step(4)
            assert joined(sv)[2] == 0
    up, on = I.radial_rupture(m.xy, 0.02, 0.1, -0.05, 0.4, 2.0, 0.0)
    with context(m) as sv:
        sv.set_bed_motion(up, on, 0.1)
        sv.set_state(s.H, s.Hu, s.Hv, 0.0)
        sv.step(4)
        assert joined(sv)[2] == 0


@pytest.mark.parametrize("n,one", [(1, True), (66, True), (300, True), (360, True)])
def test_a_callers_step_is_one_launch(n, one):
    import torch
    m = I.thacker_mesh(n=n)
    s = I.thacker_initial_state(m)
    for kw, runs in (({}, one), (dict(block_cells=192, block_threads=384), False)):
        with context(m, **kw) as sv:
            perm = torch.from_numpy(sv.permutation().astype(np.int64)).cuda()
            w = torch.empty(3, m.nc, device="cuda")
            w[:, perm] = torch.from_numpy(np.stack([s.H - m.vertex_mean(m.depth), s.Hu, s.Hv])).float().cuda()
            volna.vg_step_noalloc(sv.ctx, w.data_ptr(), torch.empty_like(w).data_ptr(), 0.0)
            assert joined(sv)[2] == (1 if runs else 0)


@pytest.mark.parametrize("dt,per_cell", [(0.0, 8 * 28 + 3), (1e-3, 8 * 24 + 3)])
def test_recordings_are_kept_by_default_only(dt, per_cell):
    m = I.thacker_mesh(n=20)
    s = I.thacker_initial_state(m)
    with context(m, 64) as sv:
        sv.set_gauges(np.array([[0.0, 0.0]]))
        sv.set_state(s.H, s.Hu, s.Hv, 0.0)
        before = sv.device_bytes()
        sv.adj_forward(8, dt, 3)
        assert sv.device_bytes() - before < 8 * m.nc * per_cell
        sv.adj_forward(8, dt, 0)
        assert sv.device_bytes() - before >= 8 * m.nc * per_cell
        sv.adj_forward(8, dt, 3)                 # a run of another shape gives them back
        assert sv.device_bytes() - before < 8 * m.nc * per_cell


def test_contexts_that_overlap():
    """Four contexts, each on a stream and a thread of its own, through launches that need
    the whole GPU and small ones, kernel graphs beside them: each result bit for bit that
    of the context alone."""
    sizes = [(32, 20), (32, 300), (64, 40), (32, 110)]
    meshes = [I.thacker_mesh(n=n) for _, n in sizes]

    def run(k, out):
        with context(meshes[k], sizes[k][0]) as sv:
            for c in (1, 40, 3, 60):
                sv.step(c)
            out[k] = sv.get_state()

    alone, together = [None] * 4, [None] * 4
    for k in range(4):
        run(k, alone)
    threads = [threading.Thread(target=run, args=(k, together)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=120)
    assert all(r is not None for r in together)
    for a, b in zip(alone, together):
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y)
