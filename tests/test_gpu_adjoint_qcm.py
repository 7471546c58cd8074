"""The void-fraction part of the adjoint (one warp per particle over the lists
of Gauss points in reach) against a brute-force sum in FP64: every degree and
both precisions, averaging spheres from half an element to lists longer than a
block of them, particles larger and smaller than the averaging sphere, at the
walls and corners, and on meshes thinner than the reach."""
import numpy as np
import pytest

from _parity import dev, host, rel_err
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu

Z = {1: [0.0, 1.0], 2: [0.0, 0.5, 1.0],
     3: [0.0, 0.5 - 0.5 / 5 ** 0.5, 0.5 + 0.5 / 5 ** 0.5, 1.0]}


def _brute(origin, h, n_el, k, lam, x, r, R):
    """sum_q w_q |J| lam(x_q) (pi a^2 / V_R) (x - x_q) / d over all Gauss points, and
    the sum of the terms' magnitudes."""
    s, w = np.polynomial.legendre.leggauss(k + 1)
    s, w = 0.5 * (s + 1), 0.5 * w
    z = Z[k]
    B = np.stack([np.prod([(s - z[b]) / (z[a] - z[b]) for b in range(k + 1) if b != a], axis=0)
                  for a in range(k + 1)], axis=-1)                       # [q, a]
    nn = [v * k + 1 for v in n_el]
    L = lam.reshape(nn[2], nn[1], nn[0])
    pts, val = [], []
    for a in range(3):
        pts.append(np.concatenate([origin[a] + h[a] * (e + s) for e in range(n_el[a])]))
    for a in range(3):                                                   # interpolate per axis
        ax = 2 - a
        blocks = [np.tensordot(L.take(range(e * k, e * k + k + 1), axis=ax), B.T, ([ax], [0]))
                  for e in range(n_el[a])]
        L = np.moveaxis(np.concatenate(blocks, axis=-1), -1, ax)
        val.append(np.tile(w, n_el[a]) * h[a])
    gq = L * val[2][:, None, None] * val[1][None, :, None] * val[0][None, None, :]
    VR = 4 / 3 * np.pi * R ** 3
    out, mag = np.zeros_like(x), np.zeros_like(x)
    for i in range(x.shape[0]):
        d = [x[i, a] - pts[a] for a in range(3)]
        d2 = d[2][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[0][None, None, :] ** 2
        dd = np.sqrt(d2)
        on = (dd < R + r[i]) & (dd > abs(R - r[i]))
        a2 = np.where(on, R * R - ((d2 - r[i] ** 2 + R * R) / (2 * np.where(on, dd, 1.0))) ** 2,
                      0.0)
        f = gq * np.pi * a2 / VR / np.where(on, dd, 1.0)
        t = [f * d[0][None, None, :], f * d[1][None, :, None], f * d[2][:, None, None]]
        out[i], mag[i] = [v.sum() for v in t], [np.abs(v).sum() for v in t]
    return out, mag


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("k,n_el,R_over_h", [
    (1, (5, 4, 6), 0.62), (2, (4, 5, 3), 0.5), (3, (3, 4, 3), 0.62),
    (1, (13, 12, 14), 4.1), (2, (1, 9, 7), 2.6), (3, (7, 2, 6), 1.9)])
def test_matches_brute_force(k, n_el, R_over_h, precision):
    import torch
    rng = np.random.default_rng(10 * k + n_el[0])
    origin, h = np.array([0.01, -0.02, 0.5]), np.array([2e-3, 2.2e-3, 1.9e-3])
    extent = h * n_el
    R = R_over_h * 2e-3
    n = 93
    x = origin + extent * rng.random((n, 3))
    x[:8] = origin + extent * np.array([[a, b, c] for a in (0, 1) for b in (0, 1) for c in (0, 1)])
    x[8:20, 0] = origin[0]
    r = R * rng.uniform(0.1, 1.9, n)
    r[20:24] = R
    nodes = int(np.prod([v * k + 1 for v in n_el]))
    lam = rng.standard_normal(nodes)
    prm = dict(synth.gas_params(1e-3, k), precision=precision, qcm_radius=R,
               cg_rtol=1e-13 if precision == 0 else 1e-12)
    zero = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda:0")  # noqa: E731
    kp = max(1, k - 1)
    pn = zero(int(np.prod([v * kp + 1 for v in n_el])))
    with cf.Context(origin, extent, n_el, k, prm) as ctx:
        g_eps, dJdx = zero(nodes), zero(n, 3)
        cf.cfdem_apply(ctx.h, dev(lam), g_eps)     # so that the adjoint solve gives lam
        eps = zero(nodes) + 0.5
        cf.cfdem_adjoint(ctx.h, n, dev(x), dev(r), zero(n, 3), zero(nodes, 3) + 0.1, pn, eps,
                         None, None, g_eps, dJdx, None)
        cf.cfdem_synchronize(ctx.h)
    want, mag = _brute(origin, h, n_el, k, lam, x, r, R)
    if precision == 0:
        assert rel_err(host(dJdx), want) <= 1e-8      # the adjoint parity tests' tolerance
    else:
        # lam changes its sign from node to node, so the terms cancel: FP32 keeps
        # each term to about ten roundings and their sum to about twenty more
        assert np.all(np.abs(host(dJdx) - want) <= 30 * 2.0 ** -24 * mag + 1e-30)
