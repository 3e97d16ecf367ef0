"""Kernels at the sizes where their split of the work can go wrong, against the
oracle or against the same call split differently."""
import numpy as np
import pytest

import oracle as O
from paper_2002_04889_gb300 import inputs as I
from paper_2002_04889_gb300 import volna

pytestmark = pytest.mark.gpu


def _moving_basin(n, half_width=1.0):
    m = I.thacker_mesh(n=n, half_width=half_width)
    s = I.thacker_initial_state(m)
    p = m.cell_points()
    deep = s.H > 2e-2
    return m, (s.H, s.Hu + 1e-3 * np.sin(3 * p[:, 0]) * deep, s.Hv + 1e-3 * np.cos(2 * p[:, 1]) * deep)


@pytest.mark.parametrize("n,n_gauges", [(7, 1), (16, 64), (16, 65), (33, 70)])
def test_adjoint_reductions_and_shared_gauge_cells(n, n_gauges):
    """CFL steps (argmin of the recorded bounds over one and several CTAs, the dot
    products of dt-bar) and gauges that share cells, one to two CTAs of gauges,
    against the oracle's taped adjoint.  FP64 sums in another order: 1e-10."""
    m, st = _moving_basin(n)
    pts = np.array([[0.0, 0.0], [0.31, -0.12], [-0.2, 0.23]])[np.arange(n_gauges) % 3]
    cells = O.OracleMesh.from_mesh(m).locate(pts)
    W = np.random.default_rng(n).normal(size=(7, n_gauges))
    with volna.Solver(64) as sv:
        sv.set_params(h_threshold=1e-5, cfl=0.9)
        sv.upload_mesh(m)
        sv.set_gauges(pts)
        sv.set_state(*st, 0.0)
        sv.adj_forward(6, 0.0)
        g = sv.adj_backward(W, m.nv)
    ad = O.ad_gauge_gradient(m, st, 0.0, 6, cells, W, h_threshold=1e-5, cfl=0.9)
    for k in ("H0", "Hu0", "Hv0", "depth"):
        b = ad["d" + k]
        assert np.linalg.norm(g[k] - b) <= 1e-10 * np.linalg.norm(b), k


@pytest.mark.parametrize("precision,n", [(64, 7), (64, 69), (64, 70), (64, 120), (64, 121), (64, 279), (32, 9), (32, 241), (32, 242)])
def test_block_shape_by_mesh_size(precision, n):
    """The block shape that the library chooses on both sides of each size at which it
    changes: FP64 equal bit for bit to blocks of 256 (the result does not depend on
    the partition), FP32 within its parity bound 1e-4 of FP64."""
    m = I.thacker_mesh(n=n, half_width=0.02 * n, h0=0.002 * n, alpha=0.02 * n, r0=0.016 * n, shuffle_cells=True)
    s = I.thacker_initial_state(m)
    p = m.cell_points() / (0.02 * n)
    st = (s.H, 0.1 * s.H * np.sin(3 * p[:, 0]), 0.1 * s.H * np.cos(2 * p[:, 1]))
    out = []
    for prec, kw in ((precision, {}), (64, dict(block_cells=256))):
        with volna.Solver(prec) as sv:
            sv.set_params(h_threshold=1e-5, cfl=0.9, **kw)
            sv.upload_mesh(m)
            sv.set_state(*st, 0.0)
            sv.step(7)
            out.append(sv.get_state())
    for a, b in zip(out[0], out[1]):
        if precision == 64:
            np.testing.assert_array_equal(a, b)
        else:
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)


@pytest.mark.parametrize("rise,t0", [(0.0, 0.0), (1e-3, 0.0), (0.02, 0.0), (0.02, 0.013), (5.0, 0.0)])
def test_moving_bed_touches_only_what_moves(rise, t0):
    """Vertices before their onset, inside their rise (some crossing both ends in one
    step, some onsets equal to a step's time), after it, and never: FP64 equal to the
    oracle's full update bit for bit, also after the motion has ended."""
    m, st = _moving_basin(20)
    r = np.hypot(m.xy[:, 0], m.xy[:, 1])
    up = 0.02 * np.exp(-(r / 0.4) ** 2) * (m.xy[:, 1] > -0.5)
    on = np.where(m.xy[:, 0] > 0.5, 1e9, np.round(0.04 * r, 3))
    prm = dict(h_threshold=1e-5, dt_fixed=0.002)
    om = O.OracleMesh.from_mesh(m)
    ref = om.run(O.params(**prm), (*st, t0), 40, bed_motion=(m.depth, up, on, rise))
    with volna.Solver(64) as sv:
        sv.set_params(**prm)
        sv.upload_mesh(m)
        sv.set_bed_motion(up, on, rise)
        sv.set_state(*st, t0)
        sv.step(40)
        got = sv.get_state()
    for a, k in zip(got, ("H", "Hu", "Hv")):
        np.testing.assert_array_equal(a, ref[k])


@pytest.mark.parametrize("n,jitter", [(8, 0.0), (33, 0.0), (40, 0.2)])
@pytest.mark.parametrize("boundary", ["wall", "open", "absorbing"])
def test_fp32_extrema_and_boundaries(n, jitter, boundary):
    """Single raised and lowered cells over water at rest (every neighbour on one side
    of the cell, increments that cancel) at and away from the boundary, on a partial
    last block: finite, and within the FP32 parity bound 1e-4 of FP64."""
    xy, tri = I.jittered_grid(n, 1.0, seed=2, jitter=jitter)
    m = I.Mesh(xy, tri, np.full(xy.shape[0], 1.0))
    H = np.ones(m.nc)
    H[::17] += 0.25
    H[5::23] -= 0.25
    st = (H, np.zeros(m.nc), np.zeros(m.nc))
    out = []
    for prec in (32, 64):
        with volna.Solver(prec) as sv:
            sv.set_params(h_threshold=1e-5, cfl=0.9)
            sv.upload_mesh(m)
            sv.set_boundary(I.boundary_edges(m, lambda p: p[:, 0] > 0.99), boundary)
            sv.set_state(*st, 0.0)
            sv.step(5)
            out.append(sv.get_state())
    for a, b in zip(*out):
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)


@pytest.mark.parametrize("every,calls", [(1, (0, 1, 2046, 3, 2047)), (3, (1, 2, 6140, 7)), (1, (5000,))])
def test_gauge_ring_over_many_calls(every, calls):
    """Records over calls of any length beside the device ring's 2048: one initial record
    and one every `every` steps, the same as a run in calls of 50 steps."""
    m, st = _moving_basin(6)
    out = []
    for parts in (calls, None):
        with volna.Solver(64) as sv:
            sv.set_params(h_threshold=1e-5, cfl=0.5, gauge_every=every)
            sv.upload_mesh(m)
            sv.set_gauges(np.array([[0.0, 0.0], [0.2, 0.1]]))
            sv.set_state(*st, 0.0)
            left = sum(calls)
            for n in parts if parts else [50] * (left // 50) + [left % 50]:
                sv.step(n)
            out.append(sv.gauges())
    assert len(out[0][0]) == 1 + sum(calls) // every
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("precision", [32, 64])
def test_run_to_several_end_times(precision):
    """t_end lives on the device: advance, plain steps past it, another end time, a new
    state and a parameter t_end, against a fresh context each time."""
    m, st = _moving_basin(12)
    def fresh(ends):
        with volna.Solver(precision) as sv:
            sv.set_params(h_threshold=1e-5, cfl=0.5)
            sv.upload_mesh(m)
            sv.set_state(*st, 0.0)
            for e in ends:
                sv.advance_to(e) if isinstance(e, float) else sv.step(e)
            return sv.get_state()
    with volna.Solver(precision) as sv:
        sv.set_params(h_threshold=1e-5, cfl=0.5)
        sv.upload_mesh(m)
        for ends in ([0.03], [0.05, 3], [4, 0.04, 0.06]):
            sv.set_state(*st, 0.0)
            for e in ends:
                sv.advance_to(e) if isinstance(e, float) else sv.step(e)
            for a, b in zip(sv.get_state(), fresh(ends)):
                np.testing.assert_array_equal(a, b)
        sv.set_params(t_end=0.02)
        sv.set_state(*st, 0.0)
        sv.step(200)
        assert sv.get_state()[3] == 0.02
        for a, b in zip(sv.get_state(), fresh([0.02])):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision,literal", [(32, 1), (64, 1), (64, 0)])
@pytest.mark.parametrize("n,steps,t_end", [(1, 2, 0.0), (9, 7, 0.0), (33, 8, 0.0), (33, 23, 0.012), (110, 9, 0.0), (290, 5, 0.0), (330, 4, 0.0), (420, 5, 0.0)])
def test_many_steps_in_one_launch(precision, literal, n, steps, t_end):
    """Steps in one launch against the step kernels one by one (which a profile asks for)
    and against a split into calls, bit for bit: state, time, counts and gauge records;
    odd and even step counts, an end time between them, meshes of one block and of more
    than one block per CTA."""
    m, st = _moving_basin(n)
    out = []
    for parts in ([steps], "profile", [1, 2, steps - 3] if steps > 3 else [0, steps]):
        with volna.Solver(precision) as sv:
            sv.set_params(h_threshold=1e-5, cfl=0.9, fp64_literal=literal, t_end=t_end, gauge_every=2)
            sv.upload_mesh(m)
            sv.set_gauges(np.array([[0.01, 0.005], [0.2, 0.1], [-0.11, 0.2]]))
            sv.set_state(*st, 0.0)
            sv.profile(parts == "profile")
            for k in [steps] if parts == "profile" else parts:
                sv.step(k)
            d = sv.diagnostics()
            out.append(list(sv.get_state()) + list(sv.gauges()) + [d[k] for k in ("t", "last_dt", "steps", "neg_count", "launches")])
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision,n,scenarios", [(32, (9, 40), (1, 5)), (32, (250, 12), (3, 8)), (64, (33, 101), (7, 2))])
def test_batch_scenario_groups(precision, n, scenarios):
    """Scenarios of a batch in groups: uneven counts (groups without a scenario), few and
    many blocks per CTA, an end time that some scenarios reach earlier; bit for bit the
    single contexts."""
    cases = [_moving_basin(k) for k in n]
    with volna.Batch(precision) as b:
        b.set_params(h_threshold=1e-5, cfl=0.9)
        for (m, st), k in zip(cases, scenarios):
            mid = b.add_mesh(m, k)
            for j in range(k):
                b.set_state(mid, j, st[0], st[1] * (1 + j), st[2], 0.0)
        b.run(0.02)
        for mid, ((m, st), k) in enumerate(zip(cases, scenarios)):
            for j in sorted({0, k - 1}):
                with volna.Solver(precision) as sv:
                    sv.set_params(h_threshold=1e-5, cfl=0.9)
                    sv.upload_mesh(m)
                    sv.set_state(st[0], st[1] * (1 + j), st[2], 0.0)
                    sv.advance_to(0.02)
                    ref = sv.get_state()
                for a, r in zip(b.get_state(mid, j)[:4], ref):
                    np.testing.assert_array_equal(a, r)


@pytest.mark.parametrize("n,t_end", [(1, 0.0), (9, 0.0), (66, 0.0), (110, 1e-3), (300, 0.0), (360, 0.0)])
def test_caller_step_in_one_launch(n, t_end):
    """The step of caller-owned states in one launch against the separate kernels (which
    a shape of 384 threads keeps), bit for bit: states, dt, past t_end, and a context of
    its own that is not disturbed; a non-finite state is reported and leaves nothing
    behind."""
    import torch
    m, st = _moving_basin(n)
    w0 = torch.from_numpy(np.stack([st[0] - m.vertex_mean(m.depth), st[1], st[2]])).float().cuda()
    out = []
    for kw in ({}, dict(block_cells=192, block_threads=384)):
        with volna.Solver(32) as sv:
            sv.set_params(h_threshold=1e-5, cfl=0.9, t_end=t_end, **kw)
            sv.upload_mesh(m)
            sv.set_state(*st, 0.0)
            sv.step(2)
            before = sv.get_state()
            w = torch.empty_like(w0)
            w[:, torch.from_numpy(sv.permutation().astype(np.int64)).cuda()] = w0
            bufs, t, res = [torch.empty_like(w) for _ in range(2)], 0.0, []
            for k in range(4):
                dt = volna.vg_step_noalloc(sv.ctx, w.data_ptr(), bufs[k & 1].data_ptr(), t)
                t, w = t + dt, bufs[k & 1]
                res += [dt, w.cpu().numpy()]
            broken = w.clone()
            broken[1, 0] = float("nan")
            broken[0, 0] += 10.0
            with pytest.raises(volna.VolnaError):
                volna.vg_step_noalloc(sv.ctx, broken.data_ptr(), bufs[0].data_ptr(), 0.0)
            res += [volna.vg_step_noalloc(sv.ctx, w.data_ptr(), bufs[0].data_ptr(), 0.0)]
            for a, b in zip(before, sv.get_state()):
                np.testing.assert_array_equal(a, b)
            out.append(res)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("dt", [0.0, 1e-3])
def test_adjoint_with_kept_recordings(dt):
    """Gradients from the forward run's own recordings (the default where they fit), from
    segments that are recomputed, and after a call that drops the recordings: bit for bit
    the same, twice in a row, and the state that the forward run leaves too."""
    m, st = _moving_basin(33)
    pts = np.array([[0.0, 0.0], [0.31, -0.12]])
    W = np.random.default_rng(5).normal(size=(12, 2))
    out = []
    with volna.Solver(64) as sv:
        sv.set_params(h_threshold=1e-5, cfl=0.9)
        sv.upload_mesh(m)
        sv.set_gauges(pts)
        for every, drop in ((0, False), (3, False), (0, True)):
            sv.set_state(*st, 0.0)
            _, eta = sv.adj_forward(11, dt, every)
            if drop:
                sv.set_params(h_threshold=1e-5, cfl=0.9)
            state = sv.get_state()
            sv.step(2)
            g, again = sv.adj_backward(W, m.nv), sv.adj_backward(W, m.nv)
            for k in g:
                np.testing.assert_array_equal(g[k], again[k])
            out.append([eta, *state] + [g[k] for k in sorted(g)])
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)
