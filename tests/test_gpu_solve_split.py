"""The FP64 solve takes its operator in double-float once the residual is below
1e-4 of the right-hand side: the true residual (with the FP64 operator) meets
the tolerance from cold and warm starts on either side of that line, and the
solution agrees with the oracle's exact solve."""
import numpy as np
import pytest

from _parity import dev, host
from oracle import oracle as O
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,n_el", [(1, (9, 8, 13)), (2, (1, 7, 12)), (2, (12, 6, 5)),
                                    (3, (5, 4, 9)), (3, (8, 1, 6))])
def test_true_residual_meets_the_tolerance(k, n_el):
    import torch
    rng = np.random.default_rng(k + n_el[0])
    origin, extent = (0.0, 0.1, -0.2), tuple(2.1e-3 * np.asarray(n_el) * (1.0, 0.9, 1.1))
    prm = dict(synth.gas_params(1.5e-3, k), cg_rtol=1e-13)
    Q = (k + 1) ** 3
    eps_q = dev(rng.uniform(0.3, 1.0, (int(np.prod(n_el)), Q)))
    nodes = int(np.prod([v * k + 1 for v in n_el]))
    z = lambda: torch.zeros(nodes, dtype=torch.float64, device="cuda:0")  # noqa: E731
    with cf.Context(origin, extent, n_el, k, prm) as ctx:
        b, y, x = z(), z(), z()
        cf.cfdem_project_rhs(ctx.h, eps_q, b)
        sol = None
        for rel in (None, 1.0, 1e-2, 3e-5, 1e-9, 0.0):
            if rel is None:
                x.zero_()
            else:
                x.copy_(sol * (1.0 + rel * dev(rng.uniform(-1, 1, nodes))))
            cf.cfdem_project(ctx.h, eps_q, x)
            cf.cfdem_synchronize(ctx.h)
            assert ctx.stats().converged == 1
            cf.cfdem_apply(ctx.h, x, y)
            torch.cuda.synchronize()
            rb = host(b)
            # the tolerance, and 50 roundings of the operator that measures it
            tol = 1e-13 + 50 * np.finfo(float).eps
            assert np.linalg.norm(rb - host(y)) <= tol * np.linalg.norm(rb)
            if sol is None:
                sol = x.clone()
        m = O.Mesh(origin, extent, n_el, k)
        ref = O.fdm_solve(m, prm["l2_smoothing"], rb)
        assert np.abs(host(sol) - ref).max() <= 1e-11 * np.abs(ref).max()
