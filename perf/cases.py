"""The work that a user of this library has it do, as cases that can be timed.

Each case goes through the public entry points of the Python binding: `Solver`
(set the state, step or advance, read the state and the gauges), the
no-allocation step, `Batch` (ensembles) and `gauge_records` (the adjoint behind
torch.autograd).  The workloads are the repository's own generators (Thacker
basin, ocean-to-coast basin, all-wet control), at sizes from an interactive toy
mesh to 4M triangles; `draw` spreads the same kinds over the whole range.

`exact` is an independent plain-torch FP64 statement of the scheme (least-squares
MUSCL with the Barth-Jespersen limiter, second-order hydrostatic reconstruction,
HLL, SSP-RK(2,2), CFL step), differentiated by autograd for the adjoint cases.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2002_04889_gb300 import inputs as I
from paper_2002_04889_gb300 import volna
from paper_2002_04889_gb300.adjoint import gauge_records

G = 9.81
CFL = 0.9
# triangles of a coast basin per (rays in angle)^2: the log-polar sector is
# ln(1000 / 50) times as long as it is wide
_XI = math.log(I.COAST_R_MAX / I.COAST_R_MIN)


# --------------------------------------------------------------------- the cases


def _case(name, kind, domain, n, **kw):
    c = dict(name=name, kind=kind, domain=domain, n=n, precision=32, literal=True, steps=0, gauges=0,
             boundary="wall", renumber="hilbert", moving_bed=False)
    c.update(kw)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # a solver inside a real-time loop that may not allocate: a small harbour
        # mesh, one call per step, the caller's own device buffers
        _case("realtime_loop_8k_fp32", "noalloc", "basin", 65, steps=8),
        # the paper's benchmark basin (about 20k triangles, three gauges) in the
        # default FP64 build that reproduces the reference solver bit for bit
        _case("basin_20k_fp64", "run", "basin", 101, precision=64, steps=100, gauges=3),
        # the same basin in FP32: calibration runs, where a step is a few launches
        _case("basin_20k_fp32", "run", "basin", 101, steps=100, gauges=3),
        # a regional forecast: ocean-to-coast basin with an absorbing offshore arc
        # and a gauge array, advanced to a given time
        _case("forecast_400k_fp32", "advance", "coast", 259, t_end=24.0, gauges=16, boundary="absorbing"),
        # the same basin driven by a kinematic rupture (the bed moves every step)
        _case("rupture_300k_fp32", "run", "coast", 223, steps=40, gauges=16, boundary="open", moving_bed=True),
        # open water everywhere: every cell reconstructs, no dry-land shortcut
        _case("allwet_1m_fp32", "run", "flat", 707, steps=40),
        # the large propagation run (the generator of the 40M-triangle benchmark)
        _case("basin_4m_fp32", "run", "basin", 1414, steps=40),
        # data assimilation through host memory: the state comes from pinned host
        # arrays, takes a few steps and goes back
        _case("host_exchange_1m_fp32", "host", "basin", 701, steps=2),
        # the coast basin in FP64, the accuracy reference of a forecast
        _case("coast_200k_fp64", "run", "coast", 183, precision=64, steps=20, gauges=16),
        # FP64 throughput build (contraction allowed)
        _case("basin_500k_fp64_contracted", "run", "basin", 499, precision=64, literal=False, steps=20),
        # uncertainty quantification: meshes of uneven size, several sources each,
        # all to a common time
        _case("ensemble_4x8_fp32", "batch", "coast", 65, meshes=4, scenarios=8, ratio=8.0, t_end=70.0, gauges=4),
        # source inversion: gauge records and their gradient with respect to the
        # initial state and the bathymetry, CFL time steps differentiated through
        _case("adjoint_50k_fp64", "adjoint", "basin", 157, precision=64, steps=40, gauges=16, dt=0.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "run", "run", "run", "run", "run", "advance", "host", "batch", "adjoint"])
    renumber = rng.choice(["hilbert", "hilbert", "hilbert", "morton", "rcm"])
    if kind == "noalloc":
        return _case(None, kind, rng.choice(["basin", "flat"]), _log(rng, 20, 355), steps=rng.randint(4, 16),
                     precision=rng.choice([32, 64]), renumber=renumber)
    if kind == "host":
        return _case(None, kind, "basin", _log(rng, 100, 1000), steps=rng.randint(1, 4), precision=rng.choice([32, 32, 64]),
                     renumber=renumber)
    if kind == "batch":
        n, meshes, scen = _log(rng, 20, 90), rng.randint(2, 5), rng.randint(2, 12)
        ratio = rng.uniform(2.0, 10.0)
        # about 120 steps of the finest mesh
        return _case(None, kind, "coast", n, meshes=meshes, scenarios=scen, ratio=round(ratio, 2),
                     t_end=round(120 * 100.0 / (n * math.sqrt(ratio)), 2), gauges=rng.randint(0, 8),
                     boundary=rng.choice(["wall", "absorbing"]))
    if kind == "adjoint":
        return _case(None, kind, "basin", _log(rng, 30, 200), precision=64, steps=rng.randint(8, 40),
                     gauges=rng.randint(1, 16), dt=rng.choice([0.0, 1.0]), boundary=rng.choice(["wall", "open", "absorbing"]))
    if kind == "advance":
        n = _log(rng, 40, 300)
        return _case(None, kind, "coast", n, t_end=round(rng.uniform(30, 90) * 100.0 / n, 2), gauges=rng.randint(0, 16),
                     boundary=rng.choice(["wall", "open", "absorbing"]), precision=rng.choice([32, 32, 64]))
    precision = rng.choice([32, 32, 64])
    domain = rng.choice(["basin", "basin", "coast", "flat"])
    n = {"basin": _log(rng, 30, 1414 if precision == 32 else 500), "coast": _log(rng, 20, 320 if precision == 32 else 180),
         "flat": _log(rng, 30, 1000 if precision == 32 else 300)}[domain]
    # a literal FP64 step costs as much as some thirty FP32 ones
    cells = _cells(dict(domain=domain, n=n))
    most = (160e6 if precision == 32 else 5e6) / cells
    return _case(None, kind, domain, n, precision=precision, literal=precision == 32 or domain == "coast" or rng.random() < 0.5,
                 steps=max(4, int(rng.uniform(0.3, 1.0) * min(most, 120))), gauges=rng.randint(0, 16) if domain != "flat" else 0,
                 boundary=rng.choice(["wall", "wall", "open", "absorbing"]) if domain == "coast" else "wall",
                 renumber=renumber, moving_bed=domain == "coast" and rng.random() < 0.3)


def _cells(case):
    n = case["n"]
    return 2 * n * int(round(_XI * n)) if case["domain"] == "coast" else 2 * n * n


def _batch_sizes(case):
    m = case["meshes"]
    return [max(8, int(round(case["n"] * math.sqrt(case["ratio"]) ** (i / (m - 1))))) for i in range(m)]


# --------------------------------------------------------------------- inputs


def _mesh(case, seed):
    n = case["n"]
    if case["domain"] == "basin":
        half = 0.5 * n * 0.04
        r0 = 0.7 + 0.2 * float(I.uniform(seed, 51, 1)[0])
        return I.thacker_mesh(n=n, half_width=half, seed=seed, h0=0.1 * half, alpha=half, r0=r0 * half, shuffle_cells=True)
    if case["domain"] == "flat":
        return I.flat_basin_mesh(n, 0.5 * n * 0.04, 10.0, seed=seed, shuffle_cells=True)
    return I.coast_mesh(n_theta=n, n_xi=int(round(_XI * n)), seed=seed)


def _state(case, mesh, seed, k=0):
    """(H, Hu, Hv) float64 numpy: the initial state of scenario k."""
    u = I.uniform(seed, 60 + k, 4)
    if case["domain"] == "coast":
        if case["moving_bed"]:
            s = I.lake_at_rest_state(mesh, 0.0)
        else:
            s = I.coast_initial_state(mesh, amplitude=1.0 + 4.0 * u[0], angle_deg=180.0 * u[1])
    elif case["domain"] == "flat":
        half = mesh.meta["half_width"]
        s = I.gaussian_hump_state(mesh, 0.0, 0.5 + u[0], half * (u[1] - 0.5), half * (u[2] - 0.5), 0.1 * half)
    else:
        s = I.thacker_initial_state(mesh)
    H, Hu, Hv = s.H, s.Hu, s.Hv
    if case["kind"] in ("noalloc", "adjoint", "host"):
        # mid-run states and generic points of the adjoint: water in motion
        p = mesh.cell_points() / np.abs(mesh.xy).max()
        c = 0.1 * H * np.sqrt(G * H)
        Hu = Hu + c * np.sin(3.0 * p[:, 0] + 2.0 * p[:, 1] + 6.0 * u[2])
        Hv = Hv + c * np.cos(2.0 * p[:, 0] - 3.0 * p[:, 1] + 6.0 * u[3])
    if case["precision"] == 32:      # what an FP32 user has in hand
        H, Hu, Hv = (a.astype(np.float32).astype(np.float64) for a in (H, Hu, Hv))
    return H, Hu, Hv


def _gauge_cells(case, mesh):
    """Gauge positions are the vertex-mean points of these cells, spread over the sea."""
    g = case["gauges"]
    if g == 0:
        return np.zeros(0, dtype=np.int64)
    wet = np.nonzero(mesh.vertex_mean(mesh.depth) > (0.3 * mesh.depth.max() if case["domain"] != "coast" else 100.0))[0]
    return wet[(np.arange(g) * 2 + 1) * len(wet) // (2 * g)]


def _threshold(case):
    return 1e-3 if case["domain"] == "coast" else 1e-5


def _boundary_edges(case, mesh):
    if case["boundary"] == "wall":
        return None
    if case["domain"] == "coast":      # the offshore arc
        return I.boundary_edges(mesh, lambda m: np.hypot(m[:, 0], m[:, 1]) > 0.99 * I.COAST_R_MAX * math.cos(0.5 / case["n"]))
    return I.boundary_edges(mesh, lambda m: m[:, 0] > 0.98 * np.abs(mesh.xy).max())


def _bed_motion(case, mesh, seed):
    u = I.uniform(seed, 70, 2)
    up, onset = I.coast_rupture(mesh, amplitude=1.0 + 4.0 * u[0], angle_deg=180.0 * u[1])
    return up, onset, 8.0


def _fixed_dt(mesh):
    """A stable fixed step of the basin: its waves cross a tenth of a square."""
    return 0.05 * mesh.meta["dx"] / math.sqrt(G * mesh.meta["h0"])


def _solver(case, mesh, seed):
    sv = volna.Solver(precision=case["precision"])
    sv.set_params(h_threshold=_threshold(case), cfl=CFL, fp64_literal=1 if case["literal"] else 0)
    sv.upload_mesh(mesh, renumber=case["renumber"])
    edges = _boundary_edges(case, mesh)
    if edges is not None:
        sv.set_boundary(edges, case["boundary"])
    if case["moving_bed"]:
        sv.set_bed_motion(*_bed_motion(case, mesh, seed))
    if case["gauges"]:
        sv.set_gauges(mesh.cell_points()[_gauge_cells(case, mesh)])
    return sv


def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    mesh = _mesh(case, seed)
    host = _state(case, mesh, seed)
    st = dict(case=case, solver=_solver(case, mesh, seed))
    dt = torch.float32 if case["precision"] == 32 else torch.float64
    if case["kind"] == "host":
        st["state"] = [torch.from_numpy(a).to(dt).pin_memory().numpy() for a in host]
        st["out"] = [torch.empty(mesh.nc, dtype=dt).pin_memory().numpy() for _ in range(3)]
    else:
        st["state"] = [torch.from_numpy(a).to(dt).cuda() for a in host]
        st["out"] = [torch.empty(mesh.nc, dtype=dt, device="cuda") for _ in range(3)]
    if case["kind"] == "noalloc":
        perm = torch.from_numpy(st["solver"].permutation().astype(np.int64)).cuda()     # new_of_old
        w = torch.from_numpy(np.stack([host[0], host[1], host[2]]))
        if case["precision"] == 32:       # row 0 of the FP32 state is the free surface
            w[0] += torch.from_numpy(-mesh.vertex_mean(mesh.depth))
        w0 = torch.empty(3, mesh.nc, dtype=dt, device="cuda")
        w0[:, perm] = w.to(dt).cuda()
        st.update(w0=w0, bufs=(torch.empty_like(w0), torch.empty_like(w0)), perm=perm)
    if case["kind"] == "adjoint":
        st["depth"] = torch.from_numpy(mesh.depth).cuda()
        st["weights"] = torch.from_numpy(_adjoint_weights(case, seed)).cuda()
        st["dt"] = _fixed_dt(mesh) if case["dt"] > 0 else 0.0
    return st


def _adjoint_weights(case, seed):
    """dJ/d(record): the residuals of a gauge misfit."""
    return 2.0 * I.uniform(seed, 80, (case["steps"] + 1) * case["gauges"]).reshape(case["steps"] + 1, -1) - 1.0


def _batch_meshes(case, seed):
    return [_mesh(dict(case, n=n), seed + 7 * i) for i, n in enumerate(_batch_sizes(case))]


def _prepare_batch(case, seed):
    b = volna.Batch(precision=32)
    b.set_params(h_threshold=_threshold(case), cfl=CFL)
    states, t0 = [], 0.0
    for i, mesh in enumerate(_batch_meshes(case, seed)):
        m = b.add_mesh(mesh, case["scenarios"])
        edges = _boundary_edges(dict(case, n=_batch_sizes(case)[i]), mesh)
        if edges is not None:
            b.set_boundary(m, edges, case["boundary"])
        if case["gauges"]:
            b.set_gauges(m, mesh.cell_points()[_gauge_cells(case, mesh)])
        states.append([_state(case, mesh, seed + 7 * i, k) for k in range(case["scenarios"])])
    return dict(case=case, batch=b, states=states, t0=t0)


# --------------------------------------------------------------------- one pass


def _records(case, t, eta):
    """An FP32 run's records are FP32 values in double arrays: kept as FP32."""
    dt = np.float32 if case["precision"] == 32 else np.float64
    return np.asarray(t, dtype=dt), np.asarray(eta, dtype=dt)


def _buffer(a, dt=np.float64):
    """A run to a given time takes a number of steps that depends on its inputs: its
    records go into a buffer of fixed length, as a monitoring program's would."""
    out = np.zeros((400,) + a.shape[1:], dtype=dt)
    out[:len(a)] = a
    return out


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        return _run_batch(st)
    sv = st["solver"]
    if kind == "noalloc":
        src, t, dts = st["w0"], 0.0, []
        for k in range(case["steps"]):
            dst = st["bufs"][k & 1]
            dt = volna.vg_step_noalloc(sv.ctx, src.data_ptr(), dst.data_ptr(), t)
            t += dt
            dts.append(dt)
            src = dst
        return dict(w=src[:, st["perm"]], dt=_records(case, dts, dts)[0])
    if kind == "adjoint":
        args = [a.clone().requires_grad_(True) for a in (*st["state"], st["depth"])]
        eta = gauge_records(sv, *args, case["steps"], st["dt"])
        grads = torch.autograd.grad(eta, args, st["weights"])
        return dict(eta=eta.detach(), H0=grads[0], Hu0=grads[1], Hv0=grads[2], depth=grads[3])
    sv.set_state(*st["state"])
    if kind == "advance":
        sv.advance_to(case["t_end"])
    else:
        sv.step(case["steps"])
    if kind == "host":
        H, Hu, Hv, t = sv.get_state(dtype=st["out"][0].dtype, out=st["out"])
        return dict(H=H, Hu=Hu, Hv=Hv, t=_records(case, t, t)[0])
    H, Hu, Hv = sv.get_state_dev(st["out"])
    res = dict(H=H, Hu=Hu, Hv=Hv)
    if case["gauges"]:
        res["gauge_t"], res["gauge_eta"] = _records(case, *sv.gauges())
        if kind == "advance":
            res["gauge_t"], res["gauge_eta"] = (_buffer(a, a.dtype) for a in (res["gauge_t"], res["gauge_eta"]))
    return res


def _run_batch(st):
    case, b = st["case"], st["batch"]
    for m, scen in enumerate(st["states"]):
        for k, s in enumerate(scen):
            b.set_state(m, k, *s, st["t0"])
    b.run(case["t_end"])
    res, times = {}, []
    for m, scen in enumerate(st["states"]):
        fields, rec_t, rec_eta = [], [], []
        for k in range(len(scen)):
            H, Hu, Hv, t, _ = b.get_state(m, k)
            fields.append(np.stack([H, Hu, Hv]))
            times.append(t)
            if case["gauges"]:
                gt, ge = b.gauges(m, k)
                rec_t.append(_buffer(gt, np.float32))
                rec_eta.append(_buffer(ge, np.float32))
        res["mesh%d" % m] = np.stack(fields).astype(np.float32)
        if case["gauges"]:
            res["gauge_t%d" % m], res["gauge_eta%d" % m] = np.stack(rec_t), np.stack(rec_eta)
    res["t"] = np.asarray(times, dtype=np.float32)
    return res


# --------------------------------------------------------------------- the work of a pass


# per cell and step: floating-point operations counted on the scheme, and the bytes of a
# compact mesh and state read and written once by each of the two stages
_FLOPS = {"basin": 509.0, "coast": 639.0, "flat": 691.0}
_BYTES = {32: 140.0, 64: 232.0}


def _finest_dt(n):
    """The coast basin's CFL step with n rays in angle, about."""
    return 100.0 / n


def work(case):
    f, by = _FLOPS[case["domain"]], _BYTES[case["precision"]]
    if case["kind"] == "batch":
        cell_steps, cells = 0.0, 0
        for n in _batch_sizes(case):
            c = _cells(dict(case, n=n)) * case["scenarios"]
            cells += c
            cell_steps += c * max(1.0, case["t_end"] / _finest_dt(n))
        return dict(bytes=by * cell_steps + 2 * 24.0 * cells, flops=f * cell_steps)
    cells = _cells(case)
    steps = case["steps"] if case["kind"] != "advance" else max(1.0, case["t_end"] / _finest_dt(case["n"]))
    if case["kind"] == "adjoint":
        # the forward run, and a reverse that costs two of it
        return dict(bytes=3.0 * by * cells * steps, flops=3.0 * f * cells * steps)
    move = 2.0 * 3.0 * (case["precision"] // 8) * cells        # the state in and out
    if case["moving_bed"]:
        by += 3.0 * case["precision"] / 8                      # the beds of every step
    return dict(bytes=by * cells * steps + move, flops=f * cells * steps)


# --------------------------------------------------------------------- the exact result


def exact(case, seed):
    """What run() returns, from a plain torch FP64 statement of the scheme."""
    if case["kind"] == "batch":
        return _exact_batch(case, seed)
    mesh = _mesh(case, seed)
    sch = _Scheme(case, mesh, _boundary_edges(case, mesh), _bed_motion(case, mesh, seed) if case["moving_bed"] else None)
    w = torch.stack([sch.t(a) for a in _state(case, mesh, seed)])[:, None, :]
    gauges = torch.as_tensor(_gauge_cells(case, mesh), device=sch.dev)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, sch, mesh, w, gauges, seed)
    t_end = case["t_end"] if case["kind"] == "advance" else 0.0
    w, t, recs, dts = sch.march(w, case["steps"] if not t_end else 10 ** 6, t_end, gauges)
    w = w[:, 0]
    if case["kind"] == "noalloc":
        if case["precision"] == 32:
            w = torch.stack([w[0] + sch.z, w[1], w[2]])
        return dict(w=w, dt=np.array([float(d) for d in dts]))
    res = dict(H=w[0], Hu=w[1], Hv=w[2])
    if case["kind"] == "host":
        return dict(res, t=np.array(float(t[0])))
    if case["gauges"]:
        res["gauge_t"] = np.array([0.0] + [float(r[0][0]) for r in recs])
        res["gauge_eta"] = torch.stack([sch.record(sch.start, gauges)[0]] + [r[1][0] for r in recs])
        if t_end:
            res["gauge_t"], res["gauge_eta"] = _buffer(res["gauge_t"]), _buffer(res["gauge_eta"].cpu().numpy())
    return res


def _exact_batch(case, seed):
    res, times = {}, []
    for m, mesh in enumerate(_batch_meshes(case, seed)):
        sub = dict(case, n=_batch_sizes(case)[m])
        sch = _Scheme(sub, mesh, _boundary_edges(sub, mesh), None)
        w = torch.stack([torch.stack([sch.t(a) for a in _state(case, mesh, seed + 7 * m, k)]) for k in range(case["scenarios"])], dim=1)
        gauges = torch.as_tensor(_gauge_cells(case, mesh), device=sch.dev)
        first = sch.record(w, gauges)
        w, t, recs, dts = sch.march(w, 10 ** 6, case["t_end"], gauges)
        res["mesh%d" % m] = w.permute(1, 0, 2)
        times += [float(x) for x in t]
        if case["gauges"]:
            moved = torch.stack(dts).cpu() > 0            # a scenario records the steps that it takes
            T, E = torch.stack([r[0] for r in recs]).cpu(), torch.stack([r[1] for r in recs]).cpu()
            rt, re = [], []
            for k in range(case["scenarios"]):
                rt.append(_buffer(torch.cat([torch.zeros(1, dtype=T.dtype), T[moved[:, k], k]]).numpy()))
                re.append(_buffer(torch.cat([first[k:k + 1].cpu(), E[moved[:, k], k]]).numpy()))
            res["gauge_t%d" % m], res["gauge_eta%d" % m] = np.stack(rt), np.stack(re)
    res["t"] = np.array(times)
    return res


def _exact_adjoint(case, sch, mesh, w, gauges, seed):
    H, Hu, Hv = (w[k, 0].clone().requires_grad_(True) for k in range(3))
    depth = sch.t(mesh.depth).requires_grad_(True)
    q = torch.stack([H, Hu, Hv])[:, None, :]
    fixed = _fixed_dt(mesh) if case["dt"] > 0 else 0.0
    sch.set_depth(depth)
    recs = [sch.record(q, gauges)[0]]
    for _ in range(case["steps"]):
        q = checkpoint(lambda x, d: sch.adjoint_step(x, d, fixed), q, depth, use_reentrant=False)
        recs.append(sch.record(q, gauges)[0])
    eta = torch.stack(recs)
    g = torch.autograd.grad(eta, (H, Hu, Hv, depth), sch.t(_adjoint_weights(case, seed)))
    return dict(eta=eta.detach(), H0=g[0], Hu0=g[1], Hv0=g[2], depth=g[3])


def _max(a, b):                    # a tie takes the first, as does its derivative
    return torch.where(a < b, b, a)


def _min(a, b):
    return torch.where(b < a, b, a)


def _pos(a):
    return torch.where(a > 0, a, torch.zeros_like(a))


def _sqrt(a):
    ok = a > 0
    return torch.where(ok, torch.sqrt(torch.where(ok, a, torch.ones_like(a))), torch.zeros_like(a))


def _over(a, b, ok):
    return torch.where(ok, a / torch.where(ok, b, torch.ones_like(b)), torch.zeros_like(a))


class _Scheme:
    """State w [3, S, nc] (H, Hu, Hv of S scenarios in the original cell order)."""

    def __init__(self, case, mesh, edges, motion):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.thr = _threshold(case)
        self.motion = None if motion is None else (self.t(motion[0]), self.t(motion[1]), motion[2])
        xy, tri = self.t(mesh.xy), torch.as_tensor(mesh.tri.astype(np.int64), device=self.dev)
        p = xy[tri]
        area2 = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1])
        tri = torch.where((area2 < 0)[:, None], tri[:, [0, 2, 1]], tri)
        first = tri.argmin(dim=1)       # local order: counter-clockwise from the smallest vertex
        tri = torch.gather(tri, 1, (first[:, None] + torch.arange(3, device=self.dev)) % 3)
        self.tri, p = tri, xy[tri]
        self.nc, self.nv = tri.shape[0], xy.shape[0]
        self.area = 0.5 * area2.abs()
        nxt = p[:, [1, 2, 0]]
        e = nxt - p
        self.len = e.norm(dim=2)
        self.nx, self.ny = e[..., 1] / self.len, -e[..., 0] / self.len
        mid, cen = 0.5 * (p + nxt), p.mean(dim=1)
        off = mid - cen[:, None]
        # faces: the two (cell, face) slots of each edge
        a, b = tri, tri[:, [1, 2, 0]]
        key = (torch.minimum(a, b) * self.nv + torch.maximum(a, b)).reshape(-1)
        key, order = torch.sort(key, stable=True)
        same = key[1:] == key[:-1]
        i = torch.nonzero(same)[:, 0]
        sL, sR = order[i], order[i + 1]
        inner = torch.zeros(3 * self.nc, dtype=torch.bool, device=self.dev)
        inner[sL] = True
        inner[sR] = True
        sB = torch.nonzero(~inner)[:, 0]
        other = torch.full((3 * self.nc,), -1, dtype=torch.int64, device=self.dev)
        other[sL], other[sR] = sR, sL
        self.kind = torch.zeros(3 * self.nc, dtype=torch.int64, device=self.dev)     # 1 wall, 2 open, 3 absorbing
        self.kind[sB] = 1
        if edges is not None:
            ed = torch.as_tensor(np.sort(edges.astype(np.int64), axis=1), device=self.dev)
            bkey = (torch.minimum(a, b) * self.nv + torch.maximum(a, b)).reshape(-1)
            hit = torch.isin(bkey, ed[:, 0] * self.nv + ed[:, 1]) & ~inner
            self.kind[hit] = 2 if case["boundary"] == "open" else 3
        # every face once: left slot, right slot (a boundary face: the left slot again)
        self.L, self.R = torch.cat([sL, sB]), torch.cat([sR, sB])
        self.bk = self.kind[self.L]
        self.slot_face = torch.empty(3 * self.nc, dtype=torch.int64, device=self.dev)
        nf = torch.arange(len(self.L), device=self.dev)
        self.slot_face[self.R] = nf
        self.slot_face[self.L] = nf
        self.right = torch.zeros(3 * self.nc, dtype=torch.bool, device=self.dev)
        self.right[sR] = True
        self.right = self.right.reshape(-1, 3)
        self.nb = torch.where(other >= 0, other // 3, torch.arange(3 * self.nc, device=self.dev) // 3).reshape(-1, 3)
        self.kind = self.kind.reshape(-1, 3)
        # least-squares weights over the neighbours' centroids (ghosts mirrored across the face)
        n = torch.stack([self.nx, self.ny], dim=2)
        d = torch.where((self.kind > 0)[..., None], 2.0 * (off * n).sum(dim=2, keepdim=True) * n, cen[self.nb] - cen[:, None])
        m = torch.einsum("kfi,kfj->kij", d, d)
        det = m[:, 0, 0] * m[:, 1, 1] - m[:, 0, 1] ** 2
        inv = torch.stack([torch.stack([m[:, 1, 1], -m[:, 0, 1]], 1), torch.stack([-m[:, 0, 1], m[:, 0, 0]], 1)], 1) / det[:, None, None]
        wts = torch.einsum("kij,kfj->kfi", inv, d)
        self.M = torch.einsum("kji,kfi->kfj", wts, off)       # increment at face f: sum_j M[f, j] (q_j - q_K)
        self.depth0 = self.t(mesh.depth)
        self.set_depth(self.depth0)
        if self.motion is not None:
            self.bed_at(torch.zeros((), dtype=torch.float64, device=self.dev))

    def t(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).to(self.dev)

    def set_depth(self, depth):
        dv = depth[self.tri]
        self.z = -dv.mean(dim=1)
        self.zf = -0.5 * (dv + dv[:, [1, 2, 0]])

    def bed_at(self, t):
        up, onset, rise = self.motion
        self.set_depth(self.depth0 - up * ((t - onset) / rise).clamp(0.0, 1.0))

    def record(self, w, gauges):
        return w[0][:, gauges] + self.z[gauges]

    def residual(self, w):
        """L(w) [3, S, nc] and max_f l_f a_f [S, nc]."""
        H = w[0]
        eta = H + self.z
        q = torch.stack([eta, w[1], w[2]])                     # [3, S, nc]
        qn = q[:, :, self.nb]                                  # [3, S, nc, 3]
        wall = self.kind == 1
        mn = w[1][..., None] * self.nx + w[2][..., None] * self.ny
        qn = torch.stack([qn[0], torch.where(wall, w[1][..., None] - 2.0 * mn * self.nx, qn[1]),
                          torch.where(wall, w[2][..., None] - 2.0 * mn * self.ny, qn[2])])
        rec = (H > self.thr) & (H[:, self.nb] > self.thr).all(dim=2)
        d = qn - q[..., None]
        D = torch.einsum("kfj,vskj->vskf", self.M, d)
        qmax = qmin = q
        for f in range(3):
            qmax, qmin = _max(qmax, qn[..., f]), _min(qmin, qn[..., f])
        alpha = torch.ones_like(q)
        for f in range(3):
            Df = D[..., f]
            r = torch.where(Df > 0, qmax - q, qmin - q)
            ok = Df != 0
            phi = torch.where(ok, _over(r, Df, ok), torch.ones_like(r))
            phi = torch.where(phi < 1, phi, torch.ones_like(phi))
            alpha = torch.where(phi < alpha, phi, alpha)
        face = q[..., None] + alpha[..., None] * D
        rec = rec & (face[0] - self.zf > self.thr).all(dim=2)
        r3 = rec[..., None]
        zs = torch.where(r3, self.zf, self.z[:, None])         # [S, nc, 3]
        Hf = torch.where(r3, face[0] - self.zf, H[..., None])
        Huf = torch.where(r3, face[1], w[1][..., None])
        Hvf = torch.where(r3, face[2], w[2][..., None])
        S = H.shape[0]
        flat = [a.reshape(S, -1) for a in (Hf, Huf, Hvf, zs)]
        hL, huL, hvL, zL = (a[:, self.L] for a in flat)
        hR, huR, hvR, zR = (a[:, self.R] for a in flat)
        nx, ny, ln = self.nx.reshape(-1)[self.L], self.ny.reshape(-1)[self.L], self.len.reshape(-1)[self.L]
        wetL, wetR = hL > self.thr, hR > self.thr
        uL, vL = _over(huL, hL, wetL), _over(hvL, hL, wetL)
        uR, vR = _over(huR, hR, wetR), _over(hvR, hR, wetR)
        unL, utL = uL * nx + vL * ny, vL * nx - uL * ny
        unR, utR = uR * nx + vR * ny, vR * nx - uR * ny
        zst = _max(zL, zR)
        sL_, sR_ = _pos(hL + zL - zst), _pos(hR + zR - zst)
        unR = torch.where(self.bk == 1, -unL, unR)
        absorb = self.bk == 3
        c0, cLf = _sqrt(G * _pos(-zL)), _sqrt(G * sL_)
        cg = _pos(0.25 * (unL + 2.0 * cLf + 2.0 * c0))
        sR_ = torch.where(absorb, cg * cg / G, sR_)
        unR = torch.where(absorb, 0.5 * (unL + 2.0 * cLf - 2.0 * c0), unR)
        # HLL in the face frame
        dryL, dryR = sL_ == 0, sR_ == 0
        cL, cR = _sqrt(G * sL_), _sqrt(G * sR_)
        us, cs = 0.5 * (unL + unR) + (cL - cR), 0.5 * (cL + cR) - 0.25 * (unR - unL)
        lo = torch.where(dryL, unR - 2.0 * cR, torch.where(dryR, unL - cL, _min(unL - cL, us - cs)))
        hi = torch.where(dryL, unR + cR, torch.where(dryR, unL + 2.0 * cL, _max(us + cs, unR + cR)))
        qL, qR = sL_ * unL, sR_ * unR
        FL = torch.stack([qL, qL * unL + 0.5 * G * sL_ * sL_, qL * utL])
        FR = torch.stack([qR, qR * unR + 0.5 * G * sR_ * sR_, qR * utR])
        dw = torch.stack([sR_ - sL_, qR - qL, sR_ * utR - sL_ * utL])
        utR_same = self.bk > 0                                  # a ghost keeps u_t
        FR = torch.where(utR_same, torch.stack([FR[0], FR[1], qR * utL]), FR)
        dw = torch.where(utR_same, torch.stack([dw[0], dw[1], (sR_ - sL_) * utL]), dw)
        midst = (lo < 0) & (hi >= 0)
        F = torch.where(lo >= 0, FL, torch.where(midst, _over(hi * FL - lo * FR + lo * hi * dw, (hi - lo).expand_as(FL), midst.expand_as(FL)), FR))
        both = dryL & dryR
        F = torch.where(both, torch.zeros_like(F), F)
        a = torch.where(hi.abs() > lo.abs(), torch.where(hi < 0, -hi, hi), torch.where(lo < 0, -lo, lo))
        a = torch.where(both, torch.zeros_like(a), a)
        Px = F[1] * nx - F[2] * ny
        Py = F[1] * ny + F[2] * nx
        PL, PR = 0.5 * G * (hL * hL - sL_ * sL_), 0.5 * G * (hR * hR - sR_ * sR_)
        tL = torch.stack([ln * F[0], ln * (Px + PL * nx), ln * (Py + PL * ny)])
        tR = torch.stack([-ln * F[0], -ln * (Px + PR * nx), -ln * (Py + PR * ny)])
        at = self.slot_face
        term = torch.where(self.right, tR[..., at].reshape(3, S, -1, 3), tL[..., at].reshape(3, S, -1, 3)).sum(dim=3)
        src = torch.where(r3, G * self.len * self.zf * (eta[..., None] - 0.5 * self.zf), torch.zeros_like(Hf))
        su, sv = (src * self.nx).sum(dim=2), (src * self.ny).sum(dim=2)
        Rr = -torch.stack([term[0], term[1] + su, term[2] + sv]) / self.area
        la = (ln * a)[:, at].reshape(S, -1, 3)
        speed = _max(_max(la[..., 0], la[..., 1]), la[..., 2])
        return Rr, speed

    def fix(self, w):
        zero = torch.zeros_like(w[0])
        H = torch.where(w[0] < 0, zero, w[0])
        wet = w[0] > self.thr
        return torch.stack([H, torch.where(wet, w[1], zero), torch.where(wet, w[2], zero)])

    def cfl_step(self, speed):
        ok = speed > 0
        bound = torch.where(ok, self.area / (3.0 * torch.where(ok, speed, torch.ones_like(speed))), torch.full_like(speed, math.inf))
        k = bound.detach().argmin(dim=1)
        return CFL * bound[torch.arange(len(k), device=self.dev), k]

    def stages(self, w, R0, dt):
        w1 = self.fix(w + dt[:, None] * R0)
        R1, _ = self.residual(w1)
        return self.fix(0.5 * w + 0.5 * (w1 + dt[:, None] * R1))

    def adjoint_step(self, w, depth, fixed):
        self.set_depth(depth)
        R0, speed = self.residual(w)
        dt = torch.full((1,), fixed, dtype=torch.float64, device=self.dev) if fixed > 0 else self.cfl_step(speed)
        return self.stages(w, R0, dt)

    def march(self, w, steps, t_end, gauges):
        self.start = w
        t = torch.zeros(w.shape[1], dtype=torch.float64, device=self.dev)
        recs, dts = [], []
        with torch.no_grad():
            for _ in range(steps):
                if t_end and bool((t >= t_end).all()):
                    break
                R0, speed = self.residual(w)
                dt = self.cfl_step(speed)
                if t_end:
                    dt = torch.where(t + dt > t_end, t_end - t, dt)
                w = self.stages(w, R0, dt)
                t = t + dt
                if self.motion is not None:
                    self.bed_at(t[0])
                dts.append(dt)
                if len(gauges):
                    recs.append((t, self.record(w, gauges)))
        return w, t, recs, dts
