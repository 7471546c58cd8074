"""The pass that splits the nodal fields into double-float once per node runs
where a kernel reads its result: many particles per node, mixed path, and no
shear force (whose kernels take the FP64 values)."""
import numpy as np
import pytest

from _parity import dev
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["forces", "adjoint", "adjoint_drag"])
@pytest.mark.parametrize("shear", [0, 1])
def test_launches_of_the_force_kernels(shear, call):
    import torch
    c = synth.make_random_case(51, n_el=(3, 3, 4), k=2, n=60, extent=(0.03, 0.03, 0.04))
    nodes = c["u_nodal"].shape[0]
    z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda:0")  # noqa: E731
    # particle-centroid scheme: the adjoint is the force kernel alone
    prm = dict(c["params"], precision=1, scheme=1, shear_force=shear)
    launches = []
    with cf.Context(c["origin"], c["extent"], c["n_el"], 2, prm) as ctx:
        for reps in (1, 40):
            x, r, up = (dev(np.tile(c[k], (reps, 1) if c[k].ndim == 2 else reps))
                        for k in ("x", "r", "u_p"))
            n = x.shape[0]
            assert (n * 27 >= 8 * nodes) == (reps == 40)
            u, p, eps, g = dev(c["u_nodal"]), dev(c["p_nodal"]), z(nodes) + 0.6, z(n, 3) + 1.0
            cf.cfdem_set_timing(ctx.h, 0)
            if call == "forces":
                cf.cfdem_forces(ctx.h, n, x, r, up, u, p, eps, z(n, 3))
            else:
                g_f = g if call == "adjoint" else None
                cf.cfdem_adjoint(ctx.h, n, x, r, up, u, p, eps, g_f, g, None, z(n, 3),
                                 z(nodes, 3))
            cf.cfdem_synchronize(ctx.h)
            launches.append(ctx.stats().kernel_launches)
    used = not shear or call == "adjoint_drag"
    assert launches[1] - launches[0] == (1 if used else 0)
