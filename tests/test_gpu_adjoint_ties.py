"""The adjoint at limiter ties: which face carries the limiter's derivative where two
faces' quotients r / D round to the same value although the D differ."""
import numpy as np
import pytest

import oracle as O
from paper_2002_04889_gb300 import inputs as I
from paper_2002_04889_gb300 import volna

pytestmark = pytest.mark.gpu


def limiter(om, K, d):
    """Increments D and quotients phi of cell K for neighbours' differences d [n][3]."""
    wx, wy, fx, fy = (om.get(k)[K] for k in ("wx", "wy", "fx", "fy"))
    gx = (wx[0] * d[:, 0] + wx[1] * d[:, 1]) + wx[2] * d[:, 2]
    gy = (wy[0] * d[:, 0] + wy[1] * d[:, 1]) + wy[2] * d[:, 2]
    D = gx[:, None] * fx + gy[:, None] * fy
    up, dn = np.maximum(0.0, d.max(axis=1)), -np.minimum(0.0, d.min(axis=1))
    return D, np.minimum(1.0, np.where(D > 0, up[:, None], dn[:, None]) / np.abs(D))


def tie(om, K, one_sign, rng):
    """Differences d of cell K whose two smallest quotients are one rounded value below 1
    at faces of different |D|, of one sign (the second of them the larger) or of two
    signs; None if it finds none."""
    def gap(d):              # zero at a tie of the asked kind; NaN where it has no sense
        D, phi = limiter(om, K, d)
        if one_sign:
            a, b = np.sort(np.abs(D) * (phi < 1), axis=1)[:, 1:].T
            i, j = np.argsort(phi, axis=1, kind="stable")[:, :2].T
            n = np.arange(len(d))
            return np.where((D[n, i] * D[n, j] > 0) & (phi[n, j] < 1), (b - a) * np.sign(j - i), np.nan)
        p, q = np.where(D > 0, phi, 1.0).min(axis=1), np.where(D < 0, phi, 1.0).min(axis=1)
        return np.where((p < 1) & (q < 1), p - q, np.nan)

    d = rng.normal(size=(20000, 3))
    if np.isnan(gap(d[:600])).all():
        return None
    f = gap(d)
    lo, hi = d[f > 0], d[f < 0]
    k = min(len(lo), len(hi))
    lo, hi = lo[:k], hi[:k]
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        over = (gap(mid) > 0)[:, None]
        lo, hi = np.where(over, mid, lo), np.where(over, hi, mid)
    n = np.arange(k)
    for _ in range(20):
        d = lo * (1 + rng.integers(-2, 3, size=lo.shape) * 2.0 ** -53)
        D, phi = limiter(om, K, d)
        i, j = np.argsort(phi, axis=1, kind="stable")[:, :2].T
        ok = (phi[n, i] == phi[n, j]) & (phi[n, i] < 1) & (phi[n, i] > 0) & ((D[n, i] * D[n, j] > 0) == one_sign)
        ok &= np.abs(D[n, j]) > np.abs(D[n, i]) if one_sign else np.abs(D[n, j]) != np.abs(D[n, i])
        if ok.any():
            return d[np.nonzero(ok)[0][0]]
    return None


@pytest.mark.filterwarnings("ignore:.*encountered in divide")
@pytest.mark.parametrize("one_sign,jitter,count", [(True, 0.2, 10), (False, 0.4, 1)])
def test_first_of_equal_quotients(one_sign, jitter, count):
    """Cells with such ties in Hu, far from one another (faces of both signs limit in a
    few badly shaped cells only), against the oracle's taped adjoint, whose minimum keeps
    the first of equals; FP64 sums in another order: 1e-10."""
    rng = np.random.default_rng(4)
    xy, tri = I.jittered_grid(24, 1.0, seed=3, jitter=jitter)
    m = I.Mesh(xy, tri, 1.0 + 0.1 * rng.random(xy.shape[0]))
    om = O.OracleMesh.from_mesh(m)
    nbr = om.get("nbr")
    Hu = np.zeros(m.nc)
    used, ties = np.zeros(m.nc, bool), []
    for K in rng.permutation(m.nc):
        near = np.unique(nbr[nbr[K]]) if (nbr[K] >= 0).all() else np.array([-1])
        if len(ties) == count or (near < 0).any() or used[near].any() or used[nbr[K]].any():
            continue
        d = tie(om, int(K), one_sign, rng)
        if d is not None:
            Hu[nbr[K]] = 2.0 ** -6 * d               # (the cell itself at rest; the scale is exact)
            used[nbr[K]] = used[near] = True
            ties.append(K)
    assert len(ties) == count
    st = (m.vertex_mean(m.depth) + 0.02 * rng.normal(size=m.nc), Hu, 0.05 * rng.normal(size=m.nc))
    cells = np.unique(np.concatenate([[K, *nbr[K]] for K in ties]))
    pts = np.array([xy[tri[c]].mean(axis=0) for c in cells])
    W = rng.normal(size=(2, len(cells)))
    with volna.Solver(64) as sv:
        sv.set_params(h_threshold=1e-5, cfl=0.9)
        sv.upload_mesh(m)
        sv.set_gauges(pts)
        sv.set_state(*st, 0.0)
        sv.adj_forward(1, 1e-3)
        g = sv.adj_backward(W, m.nv)
    ad = O.ad_gauge_gradient(m, st, 1e-3, 1, om.locate(pts), W, h_threshold=1e-5)
    for k in ("H0", "Hu0", "Hv0", "depth"):
        b = ad["d" + k]
        assert np.linalg.norm(g[k] - b) <= 1e-10 * np.linalg.norm(b), k
