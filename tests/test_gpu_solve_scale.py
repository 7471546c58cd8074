"""The FP64 solve does not depend on the size of its right-hand side: the
projection of a scaled field and the adjoint of scaled seeds take the same
iterations and give the scaled results, from sizes that a mean over many
particles brings about up to very large ones."""
import numpy as np
import pytest

from _parity import dev, host
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,n_el", [(1, (9, 8, 13)), (2, (12, 6, 5)), (3, (5, 4, 9))])
@pytest.mark.parametrize("h", [3.5e-3, 20.0])
def test_projection_of_a_scaled_field(k, n_el, h):
    import torch
    rng = np.random.default_rng(3)
    prm = dict(synth.gas_params(0.5 * h, k), cg_rtol=1e-13, l2_smoothing=(0.3 * h) ** 2)
    eps_q = rng.uniform(0.3, 1.0, (int(np.prod(n_el)), (k + 1) ** 3))
    nodes = int(np.prod([v * k + 1 for v in n_el]))
    first = None
    with cf.Context((0, 0, 0), tuple(h * np.asarray(n_el)), n_el, k, prm) as ctx:
        for e in (0, -10, -20, -30, -40, -50, -60, 30, 60):
            x = torch.zeros(nodes, dtype=torch.float64, device="cuda:0")
            cf.cfdem_project(ctx.h, dev(eps_q * 2.0 ** e), x)
            cf.cfdem_synchronize(ctx.h)
            s = ctx.stats()
            got = host(x) * 2.0 ** -e
            if first is None:
                first = (got, s.cg_iterations)
            assert s.converged == 1 and s.cg_iterations == first[1]
            # both meet a residual of 1e-13 of b (condition number below 100)
            assert np.abs(got - first[0]).max() <= 1e-11 * np.abs(first[0]).max()


@pytest.mark.parametrize("k", [1, 2, 3])
def test_adjoint_of_scaled_seeds(k):
    import torch
    c = synth.make_random_case(21 + k, n_el=(4, 5, 3), k=k, n=80, extent=(0.04, 0.05, 0.03))
    rng = np.random.default_rng(k)
    n, nodes = c["x"].shape[0], c["u_nodal"].shape[0]
    t = [dev(c[v]) for v in ("x", "r", "u_p", "u_nodal", "p_nodal")]
    eps = dev(rng.uniform(0.5, 0.8, nodes))
    seed = rng.standard_normal((n, 3))
    first = None
    with cf.Context(c["origin"], c["extent"], c["n_el"], k,
                    dict(c["params"], cg_rtol=1e-13)) as ctx:
        for e in (0, -13, -27, -40):
            dJdx = torch.zeros((n, 3), dtype=torch.float64, device="cuda:0")
            dJdu = torch.zeros((nodes, 3), dtype=torch.float64, device="cuda:0")
            cf.cfdem_adjoint(ctx.h, n, *t, eps, None, dev(seed * 2.0 ** e), None, dJdx, dJdu)
            cf.cfdem_synchronize(ctx.h)
            assert ctx.stats().converged == 1
            got = [host(v) * 2.0 ** -e for v in (dJdx, dJdu)]
            first = first or got
            for a, b in zip(got, first):
                assert np.abs(a - b).max() <= 1e-11 * np.abs(b).max()
