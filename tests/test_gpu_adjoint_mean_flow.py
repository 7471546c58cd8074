"""The mixed path's force adjoint in a flow with a large mean velocity: the
drag depends on the slip, so a velocity added to fluid and particles alike
leaves the gradients as they are, and the interpolation has to cancel it to
double-float and not to FP32 accuracy."""
import numpy as np
import pytest

from _parity import dev, host
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 2000])   # nodal values split per particle, per node
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("mean", [0.0, 1e2, 1e5])
def test_gradients_do_not_lose_the_variation(k, n, mean):
    import torch
    c = synth.make_random_case(40 + k, n_el=(4, 5, 3), k=k, n=40, extent=(0.04, 0.05, 0.03))
    rng = np.random.default_rng(k)
    reps = n // 40
    x, r = np.tile(c["x"], (reps, 1)), np.tile(c["r"], reps)   # forces see one particle each
    shift = mean * np.array([1.0, 0.3, -0.5])
    u, up = c["u_nodal"] + shift, np.tile(c["u_p"], (reps, 1)) + shift
    nodes = u.shape[0]
    assert (n * (k + 1) ** 3 >= 8 * nodes) == (n == 2000)
    eps = rng.uniform(0.5, 0.7, nodes)
    g_f, g_fd = rng.standard_normal((n, 3)), rng.standard_normal((n, 3))
    got = []
    for precision in (0, 1):
        dJdx = torch.zeros((n, 3), dtype=torch.float64, device="cuda:0")
        dJdu = torch.zeros((nodes, 3), dtype=torch.float64, device="cuda:0")
        with cf.Context(c["origin"], c["extent"], c["n_el"], k,
                        dict(c["params"], precision=precision)) as ctx:
            cf.cfdem_adjoint(ctx.h, n, dev(x), dev(r), dev(up), dev(u), dev(c["p_nodal"]),
                             dev(eps), dev(g_f), dev(g_fd), None, dJdx, dJdu)
            cf.cfdem_synchronize(ctx.h)
        got.append((host(dJdx), host(dJdu)))
    # the closure's derivatives, about 30 FP32 operations deep; double-float's
    # share of the mean is 1e5 x 2^-45
    for a, b in zip(*got):
        assert np.linalg.norm(a - b) <= 32 * 2.0 ** -24 * np.linalg.norm(a)
