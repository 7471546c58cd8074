"""Location on curved meshes where coordinates do not resolve the reference
coordinates to the iteration's 1e-13 -- far from the origin -- and on meshes of
sizes near the ends of FP32's exponents: the elements are the definition's,
points that its FP64 iteration does not find included."""
import numpy as np
import pytest

from _parity import dev, host
from oracle import oracle as O
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


def _mesh(k):
    m = synth.make_box_mapped_mesh((0, 0, 0), (3.0, 4.0, 2.0), (3, 4, 2), k)
    x, y, z = m["nodes"].T
    bent = np.stack([x + 0.1 * np.sin(1.1 * y + 0.4) * np.cos(0.7 * z),
                     y + 0.1 * np.sin(0.9 * z + 0.8 * x),
                     z + 0.1 * np.cos(0.8 * x + 0.3) * np.sin(1.3 * y)], axis=1)
    return m["conn"], bent


def _locate(k, conn, nodes, x):
    import torch
    n = x.shape[0]
    with cf.MappedMesh(k, conn, nodes) as mm:
        elem = torch.zeros(n, dtype=torch.int32, device="cuda:0")
        xi = torch.zeros((n, 3), dtype=torch.float64, device="cuda:0")
        assert mm.locate(n, dev(x), elem, xi) == cf.OK
        torch.cuda.synchronize()
    return host(elem), host(xi)


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("shift", [100.0, 300.0, -1e3, 1e4, 1e7])
def test_far_meshes_follow_the_definition(k, shift):
    conn, bent = _mesh(k)
    nodes = np.ascontiguousarray(bent + shift * np.array([1.0, 0.7, -1.1]))
    rng = np.random.default_rng(k)
    x = nodes.min(0) + (nodes.max(0) - nodes.min(0)) * rng.random((3001, 3))
    e_ref, xi_ref, miss = O.locate_mapped(k, conn, nodes, x)
    elem, xi = _locate(k, conn, nodes, x)
    assert np.array_equal(elem, e_ref)
    assert np.array_equal(xi, xi_ref)          # the same arithmetic
    assert (miss > 1000) == (abs(shift) >= 1e3)


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("shift", [0.0, 5.0, 10.0, 20.0, 40.0])
def test_meshes_about_the_line(k, shift):
    """Distances on either side of the one from which the definition's own
    iteration decides (64 roundings of the coordinates)."""
    conn, bent = _mesh(k)
    nodes = np.ascontiguousarray(bent + shift)
    rng = np.random.default_rng(10 + k)
    x = nodes.min(0) + (nodes.max(0) - nodes.min(0)) * rng.random((3001, 3))
    e_ref, xi_ref, _ = O.locate_mapped(k, conn, nodes, x)
    elem, xi = _locate(k, conn, nodes, x)
    assert np.array_equal(elem, e_ref)
    assert np.abs(xi - xi_ref).max() <= 1e-12 + 64 * 2.0 ** -52 * np.abs(nodes).max()


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("scale", [1e-45, 1e-39, 1e-30, 1e-21, 1e-19, 1e19, 1e21, 1e40])
def test_tiny_and_huge_meshes(k, scale):
    conn, bent = _mesh(k)
    nodes = np.ascontiguousarray(bent * scale)
    rng = np.random.default_rng(20 + k)
    x = rng.random((1500, 3)) * np.array([3.0, 4.0, 2.0]) * scale
    e_ref, xi_ref, _ = O.locate_mapped(k, conn, nodes, x)
    elem, xi = _locate(k, conn, nodes, x)
    assert np.array_equal(elem, e_ref)
    assert np.abs(xi - xi_ref).max() <= 1e-12
