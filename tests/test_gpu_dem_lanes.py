"""The DEM kernel's eight lanes per particle where they can go wrong, against
the FP64 oracle: particle counts around the lane groups and blocks, cell grids
of one cell, of long rows and of rows that straddle the ranges' tiles, more
screened candidates than the list holds, and contacts that open and close."""
import numpy as np
import pytest

from _parity import dev, host, rel_err
from oracle import dem as D
from paper_2211_01185_gb300 import cfdem as cf

pytestmark = pytest.mark.gpu


def _run(x, v, w, r, p, dt, nsub, precision, capacity=24):
    prm = {k: p[k] for k in D.PARAM_KEYS}
    prm.update(g=p["g"], lo=p["lo"], hi=p["hi"], max_radius=float(r.max()), capacity=capacity,
               precision=precision)
    tx, tv, tw = dev(x), dev(v), dev(w)
    with cf.Dem(prm) as dm:
        for k in nsub:
            dm.step(tx, tv, tw, dev(r), None, dt, k)
        assert dm.synchronize() == cf.OK, dm.last_error()
    ref = D.State(x, v, w, r, capacity=capacity)
    for k in nsub:
        assert ref.step(p, dt, k) == 0
    # FP64: the parity tests' metric and tolerance.  Mixed: the FP32 contact
    # arithmetic (about ten roundings of 6e-8 a force, and the contacts' own
    # cancellation) in the 2-norm; per component the rounding of small
    # differences says nothing (the same inputs give 1e-6 to 8e-5 there)
    for got, new, old in ((tx, ref.x, x), (tv, ref.v, v), (tw, ref.w, w)):
        if precision == 0:
            assert rel_err(host(got) - old, new - old) <= 1e-9
        else:
            assert np.linalg.norm(host(got) - new) <= 1e-6 * np.linalg.norm(new - old)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,side", [(1, 1), (15, 3), (16, 3), (17, 1), (129, 5), (300, 2)])
def test_counts_and_columns(n, side, precision):
    """A slightly compressed column of side x side spheres, numbered at random,
    that rests on the floor and the walls and flies apart."""
    rng = np.random.default_rng(n)
    r = rng.uniform(0.9e-3, 1.0e-3, n)
    k = np.arange(n)
    site = np.stack([k % side, k // side % side, k // (side * side)], axis=1)
    x = 0.95e-3 + 1.88e-3 * site + 1e-5 * rng.standard_normal((n, 3))
    perm = rng.permutation(n)
    x, r = np.ascontiguousarray(x[perm]), r[perm]
    hi = 1.9e-3 + 1.88e-3 * site.max(0) + [0, 0, 2e-3]
    p = D.glass_params((0, 0, 0), tuple(hi), rolling_friction=0.02, wall_rolling_friction=0.01)
    v, w = 0.05 * rng.standard_normal((n, 3)), 20.0 * rng.standard_normal((n, 3))
    _run(x, v, w, r, p, 2e-6, [7, 12], precision)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_long_rows(axis, precision):
    """A chain of touching spheres along one axis of a box of ~1500 cells: rows
    longer than half a tile of the ranges, and many short rows."""
    n = 1200
    rng = np.random.default_rng(axis)
    r = np.full(n, 1e-3)
    x = np.full((n, 3), 1.5e-3)
    x[:, axis] = 1e-3 + 1.99e-3 * np.arange(n)
    hi = np.full(3, 6e-3)
    hi[axis] = 3.0
    p = D.glass_params((0, 0, 0), tuple(hi))
    v, w = 0.02 * rng.standard_normal((n, 3)), 10.0 * rng.standard_normal((n, 3))
    _run(x, v, w, r, p, 2e-6, [9], precision)


@pytest.mark.parametrize("precision", [0, 1])
def test_more_screened_than_listed(precision):
    """50 spheres touch the large one and 40 miss it by less than the screen's
    margin: 90 screened candidates, 50 contacts."""
    k = np.arange(90) + 0.5
    phi, th = np.arccos(1 - 2 * k / 90), np.pi * (1 + 5 ** 0.5) * k
    u = np.stack([np.cos(th) * np.sin(phi), np.sin(th) * np.sin(phi), np.cos(phi)], axis=1)
    gap = np.where(np.arange(90) % 9 < 5, -2e-6, 1e-8)
    c = np.array([0.01, 0.01, 0.01])
    x = np.vstack([c, c + (1.15e-3 + gap)[:, None] * u])
    r = np.concatenate([[1e-3], np.full(90, 0.15e-3)])
    rng = np.random.default_rng(9)
    w = 5.0 * rng.standard_normal(x.shape)
    p = D.glass_params((0, 0, 0), (0.02, 0.02, 0.02), g=(0.0, 0.0, 0.0))
    # no relative approach within the sub-steps: the misses stay misses
    v = np.zeros_like(x)
    v[1:] = 1e-6 * u
    _run(x, v, w, r, p, 1e-8, [2], precision, capacity=64)
