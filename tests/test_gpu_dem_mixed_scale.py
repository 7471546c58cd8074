"""The mixed DEM path's contact test and overlaps are FP64: its forces keep FP32
accuracy in boxes that are thousands of radii long and at overlaps of a
millionth of the radius, and for particles down to nanometres; against the FP64
path on the same isolated pairs and wall contacts."""
import numpy as np
import pytest

from _parity import dev, host
from oracle import dem as D
from paper_2211_01185_gb300 import cfdem as cf

pytestmark = pytest.mark.gpu


def _kick(x, r, box, precision, dt, v, max_radius):
    """velocity change of one sub-step"""
    p = D.glass_params((0, 0, 0), tuple(box), g=(0, 0, 0), friction=0.0, wall_friction=0.0)
    prm = {k: p[k] for k in D.PARAM_KEYS}
    prm.update(g=p["g"], lo=p["lo"], hi=p["hi"], max_radius=max_radius, capacity=24,
               precision=precision)
    tx, tv, tw = dev(x), dev(v), dev(np.zeros_like(x))
    with cf.Dem(prm) as dm:
        dm.step(tx, tv, tw, dev(r), None, dt, 1)
        assert dm.synchronize() == cf.OK, dm.last_error()
    return host(tv) - v


def _compare(x, r, box, dt, v=None, max_radius=None):
    v = np.zeros_like(x) if v is None else v
    max_radius = max_radius or float(r.max())
    a, b = (_kick(x, r, box, p, dt, v, max_radius) for p in (0, 1))
    size = np.linalg.norm(a, axis=1)
    assert (size > 0).sum() > 0.9 * len(x)
    assert np.array_equal(size > 0, np.linalg.norm(b, axis=1) > 0)
    hit = size > 0
    # a force is about 30 FP32 operations deep; a sub-step moves the particles
    # by less than 1e-9 of the smallest overlap
    assert (np.linalg.norm(a - b, axis=1)[hit] <= 40 * 2.0 ** -24 * size[hit]).all()


@pytest.mark.parametrize("length,overlap", [(20, 1e-3), (2e3, 1e-4), (2e3, 1e-6), (8e3, 1e-5),
                                            (8e3, 1e-7)])
def test_pairs_in_long_boxes(length, overlap):
    rng = np.random.default_rng(int(length))
    rad, n = 1e-3, 400
    box = rad * np.array([length, 20.0, 20.0])
    r = np.full(2 * n, rad)
    # pairs on a lattice along the box, so that they do not meet one another
    k = np.arange(n)
    c = np.stack([(k + 0.5) / n * 0.9 * length + 0.02 * length, np.full(n, 5.0), np.full(n, 5.0)],
                 axis=1)
    c[:, 1] += 10.0 * (k % 2)
    c[:, 2] += 10.0 * (k // 2 % 2)
    u = rng.standard_normal((n, 3)) * [0.05, 1.0, 1.0]
    u /= np.linalg.norm(u, axis=1)[:, None]
    d = 2.0 * (1.0 - overlap * rng.uniform(0.1, 1.0, n))
    if length < 100:
        c, u, d, r = c[:8], u[:8], d[:8], r[:16]
        c[:, 0] = 2.0 + 2.0 * np.arange(8) % 16
    x = np.empty((2 * len(c), 3))
    x[0::2], x[1::2] = c, c + d[:, None] * u
    _compare(rad * x, r, box, 1e-16)


@pytest.mark.parametrize("overlap", [1e-3, 1e-6])
def test_walls_of_long_boxes(overlap):
    rng = np.random.default_rng(5)
    rad = 1e-3
    box = rad * np.array([20.0, 20.0, 6e3])
    n = 300
    x = np.full((n, 3), 10.0 * rad)
    x[:, 2] = (3.0 + 19.0 * np.arange(n)) * rad
    gap = rad * (1.0 - overlap * rng.uniform(0.1, 1.0, n))
    x[0::2, 0], x[1::2, 0] = gap[0::2], box[0] - gap[1::2]
    x[-1] = [10.0 * rad, 10.0 * rad, box[2] - gap[-1]]
    _compare(x, np.full(n, rad), box, 1e-16)


@pytest.mark.parametrize("stated", [1.0, 1e7])
@pytest.mark.parametrize("rad", [1e-2, 1e-5, 1e-7, 1e-8, 2e-9])
def test_particle_sizes(rad, stated):
    """With a relative velocity, so that the damping (root of the effective
    mass) is in the forces; also with a stated largest radius far above the
    particles' own."""
    rng = np.random.default_rng(6)
    n = 100
    c = np.stack([4.0 + 5.0 * np.arange(n), np.full(n, 10.0), np.full(n, 10.0)], axis=1)
    u = rng.standard_normal((n, 3)) * [0.05, 1.0, 1.0]
    u /= np.linalg.norm(u, axis=1)[:, None]
    x = np.empty((2 * n, 3))
    x[0::2] = c
    x[1::2] = c + (2.0 - 2e-2 * rng.uniform(0.5, 1.0, n))[:, None] * u
    v = np.zeros_like(x)
    v[1::2] = -0.3 * u
    box = rad * np.array([5.0 * n + 10.0, 20.0, 20.0])
    _compare(rad * x, np.full(2 * n, rad), box, 1e-12 * rad, v, stated * rad)
