"""The FP32 screen of the mapped location (candidates thrown out or started in
FP32, finished with FP64 residuals) against the oracle's plain FP64 Newton
inversion where the screen's decisions are closest: points on, just inside and
just outside element faces, strongly distorted elements, a mesh far from the
origin and a tiny one; and the interpolation over every component count."""
import numpy as np
import pytest

from _parity import dev, host
from oracle import oracle as O
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu

Z = {1: [0.0, 1.0], 2: [0.0, 0.5, 1.0],
     3: [0.0, 0.5 - 0.5 / 5 ** 0.5, 0.5 + 0.5 / 5 ** 0.5, 1.0]}


def _basis(k, t):
    z = Z[k]
    return np.stack([np.prod([(t - z[b]) / (z[a] - z[b]) for b in range(k + 1) if b != a], axis=0)
                     for a in range(k + 1)], axis=-1)


def _mesh(k, scale, shift, bend):
    """A 3 x 4 x 2 box of unit elements, bent by a smooth map, scaled and shifted."""
    m = synth.make_box_mapped_mesh((0, 0, 0), (3.0, 4.0, 2.0), (3, 4, 2), k)
    x, y, z = m["nodes"].T
    bent = np.stack([x + bend * np.sin(1.1 * y + 0.4) * np.cos(0.7 * z),
                     y + bend * np.sin(0.9 * z + 0.8 * x),
                     z + bend * np.cos(0.8 * x + 0.3) * np.sin(1.3 * y)], axis=1)
    return m["conn"], np.ascontiguousarray(scale * bent + shift)


def _points(rng, k, conn, nodes, n):
    """Points at chosen reference coordinates, some of them at faces (on them
    and 1e-12 to 2e-2 to either side), and a cloud around the mesh."""
    xi = rng.random((n, 3))
    off = np.array([0.0, 1e-12, -1e-12, 1e-6, -1e-6, 1e-3, -1e-3, 9e-3, 1.1e-2, 2e-2])
    face = rng.random((n, 3)) < 0.4
    near = rng.integers(0, 2, (n, 3)) + rng.choice(off, (n, 3))
    xi = np.where(face, near, xi)
    e = rng.integers(0, conn.shape[0], n)
    P = nodes[conn[e]].reshape(n, k + 1, k + 1, k + 1, 3)
    x = np.einsum("nc,nb,na,ncbai->ni", _basis(k, xi[:, 2]), _basis(k, xi[:, 1]),
                  _basis(k, xi[:, 0]), P)
    lo, hi = nodes.min(0), nodes.max(0)
    cloud = lo + (hi - lo) * (1.2 * rng.random((n, 3)) - 0.1)
    return np.concatenate([x, cloud])


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("scale,shift,bend", [(1.0, 0.0, 0.0), (1e-3, 0.0, 0.12),
                                              (1.0, 30.0, 0.2), (1e-7, 0.0, 0.3)])
def test_screened_location_matches_oracle(k, scale, shift, bend):
    conn, nodes = _mesh(k, scale, shift, bend)
    rng = np.random.default_rng(100 * k + int(10 * bend))
    x = _points(rng, k, conn, nodes, 3001)
    e_ref, xi_ref, miss = O.locate_mapped(k, conn, nodes, x)
    assert 0 < miss < x.shape[0]
    n = x.shape[0]
    import torch
    with cf.MappedMesh(k, conn, nodes) as mm:
        elem = torch.zeros(n, dtype=torch.int32, device="cuda:0")
        xi = torch.zeros((n, 3), dtype=torch.float64, device="cuda:0")
        assert mm.locate(n, dev(x), elem, xi) == cf.OK
        torch.cuda.synchronize()
    assert np.array_equal(host(elem), e_ref)
    # the step criterion, and what coordinates of this size resolve of xi
    tol = 1e-12 + 64 * np.finfo(float).eps * np.abs(nodes).max() / scale
    assert np.allclose(host(xi), xi_ref, rtol=0, atol=tol)


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("ncomp", [1, 3, 4, 5, 8])
def test_interpolation_of_any_component_count(k, ncomp):
    import torch
    conn, nodes = _mesh(k, 1.0, 0.0, 0.1)
    rng = np.random.default_rng(7 + ncomp)
    n = 515
    e = rng.integers(-1, conn.shape[0], n).astype(np.int32)
    xi = rng.random((n, 3))
    field = rng.standard_normal((nodes.shape[0], ncomp))
    F = field[conn[e]].reshape(n, k + 1, k + 1, k + 1, ncomp)
    want = np.einsum("nc,nb,na,ncbaj->nj", _basis(k, xi[:, 2]), _basis(k, xi[:, 1]),
                     _basis(k, xi[:, 0]), F)
    want[e < 0] = 0.0
    with cf.MappedMesh(k, conn, nodes) as mm:
        out = torch.full((n, ncomp), 7.0, dtype=torch.float64, device="cuda:0")
        ed = torch.as_tensor(e, device="cuda:0")
        assert mm.interpolate(n, ed, dev(xi), ncomp, dev(field), out) == cf.OK
        torch.cuda.synchronize()
    # (k + 1)^3 products of at most ~3 rounding errors each, |l| sums below 5
    assert np.allclose(host(out), want, rtol=0, atol=64 * 3 * 5 * np.finfo(float).eps * 4)
