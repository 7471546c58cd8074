"""The FP64 void fraction (groups of 32 candidates against the element's Gauss
points, hits summed by a few lanes per point) against a brute-force sum in
FP64: every degree, candidate counts around the size of a group, every pair a
hit and few hits, particles inside the averaging sphere, larger than it and
centred on a Gauss point, with and without the volume-conserving scale."""
import numpy as np
import pytest

from _parity import dev, host
from oracle import oracle as O
from paper_2211_01185_gb300 import cfdem as cf

pytestmark = pytest.mark.gpu


def _brute(m, R, x, r):
    """Per Gauss point: void fraction, neighbours, sum of their ids, error bound."""
    g, _ = O.gauss_rule(m.nq)
    ax = [m.origin[a] + m.h[a] * (np.arange(m.n_el[a])[:, None] + g) for a in range(3)]
    # [ez, ey, ex, qz, qy, qx]
    Z, Y, X = (np.broadcast_to(ax[2][:, None, None, :, None, None],
                               (*m.n_el[::-1], m.nq, m.nq, m.nq)),
               ax[1][None, :, None, None, :, None], ax[0][None, None, :, None, None, :])
    vr = 4.0 / 3.0 * np.pi * R ** 3
    s, c, ids, bound = (np.zeros(Z.shape) for _ in range(4))
    for i in range(x.shape[0]):
        d2 = (x[i, 0] - X) ** 2 + (x[i, 1] - Y) ** 2 + (x[i, 2] - Z) ** 2
        hit = d2 < (R + r[i]) ** 2
        d = np.sqrt(d2)
        dm, mn = abs(R - r[i]), min(R, r[i])
        full = 4.0 / 3.0 * np.pi * mn ** 3
        dd = np.where(d > dm, d, 1.0)
        lens = np.pi / 12 * (R + r[i] - dd) ** 2 * (dd * dd + 2 * dd * (R + r[i]) - 3 * dm * dm) / dd
        s += np.where(hit, np.where(d > dm, lens, full), 0.0)
        c += hit
        ids += hit * i
        # double-float arithmetic (2^-48 per rounding): 2^-42 of the smaller
        # sphere per hit for the products and sums, and R + r - d known to
        # 2^-44 of the box (the positions) plus R + r (d and the radii) moves
        # the lens by its open area, at most pi min(R, r)^2
        bound += hit * (2.0 ** -42 * full / vr +
                        2.0 ** -44 * (np.max(m.extent) + R + r[i]) * np.pi * mn ** 2 / vr)
    sh = (m.n_elem, m.Q)
    return (1.0 - s / vr).reshape(sh), c.reshape(sh), ids.reshape(sh), bound.reshape(sh) + 2.0 ** -50


@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 200])
@pytest.mark.parametrize("k,n_el,R_over_h", [
    (1, (3, 2, 2), 0.6), (2, (2, 3, 2), 0.4), (3, (2, 1, 3), 0.6),
    (1, (2, 2, 1), 3.0), (2, (1, 2, 2), 2.5), (3, (1, 1, 2), 2.5)])
def test_matches_brute_force(k, n_el, R_over_h, n):
    import torch
    rng = np.random.default_rng(100 * k + n)
    h = np.array([0.9e-2, 1e-2, 1.1e-2])
    origin, extent = np.array([-0.3, 0.1, 0.02]), h * n_el
    m = O.Mesh(origin, extent, n_el, k)
    R = R_over_h * 1e-2
    x = origin + rng.uniform(size=(n, 3)) * extent
    r = R * 10.0 ** rng.uniform(-1.5, 0.3, n)
    g, _ = O.gauss_rule(m.nq)
    x[0] = origin + h * g[0]  # on a Gauss point
    r[n // 2] = R             # no core inside the averaging sphere
    prm = dict(precision=0, qcm_radius=R)
    with cf.Context(origin, extent, n_el, k, prm) as ctx:
        eps = torch.zeros((m.n_elem, m.Q), dtype=torch.float64, device="cuda:0")
        cnt = torch.zeros((m.n_elem, m.Q), dtype=torch.int32, device="cuda:0")
        ids = torch.zeros((m.n_elem, m.Q), dtype=torch.int64, device="cuda:0")
        bare = torch.zeros_like(eps)
        cf.cfdem_void_fraction(ctx.h, n, dev(x), dev(r), eps, cnt, ids)
        cf.cfdem_void_fraction(ctx.h, n, dev(x), dev(r), bare, None, None)
        cf.cfdem_synchronize(ctx.h)
    e_ref, c_ref, i_ref, bound = _brute(m, R, x, r)
    assert np.array_equal(host(cnt), c_ref.astype(np.int64))
    assert np.array_equal(host(ids), i_ref.astype(np.int64))
    assert np.max(np.abs(host(eps) - e_ref) / bound) <= 1.0
    assert np.array_equal(host(bare), host(eps))
    with cf.Context(origin, extent, n_el, k, dict(prm, qcm_conserve=1)) as ctx:
        cf.cfdem_void_fraction(ctx.h, n, dev(x), dev(r), eps, cnt, ids)
        cf.cfdem_synchronize(ctx.h)
    assert np.array_equal(host(cnt), c_ref.astype(np.int64))
    e_con, _, _ = O.qcm(m, R, x, r, conserve=True)
    assert np.max(np.abs(host(eps) - e_con) / np.maximum(np.abs(e_con), 1e-3 * np.max(np.abs(e_con)))) <= 1e-10
