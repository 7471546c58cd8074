"""kernel_launches counts the kernels of an eager step whether its solve runs
launch by launch or as the context's graph."""
import pytest

from _parity import dev
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_steps_count_alike(k, precision):
    import torch
    c = synth.make_random_case(61 + k, n_el=(4, 5, 6), k=k, n=150, extent=(0.04, 0.05, 0.06))
    n = c["x"].shape[0]
    t = [dev(c[v]) for v in ("x", "r", "u_p", "u_nodal", "p_nodal")]
    eps = torch.zeros(c["u_nodal"].shape[0], dtype=torch.float64, device="cuda:0")
    f = torch.zeros((n, 3), dtype=torch.float64, device="cuda:0")
    counts = []
    with cf.Context(c["origin"], c["extent"], c["n_el"], k,
                    dict(c["params"], precision=precision, cg_rtol=1e-12, autotune=0)) as ctx:
        for rep in range(5):
            eps.zero_()
            before = ctx.stats().kernel_launches
            cf.cfdem_coupling_step(ctx.h, n, *t, eps, f)
            counts.append(ctx.stats().kernel_launches - before)
            cf.cfdem_synchronize(ctx.h)
    # the graph has the condition of its loop on top, and the launches queued
    # ahead of it are those of the first chunk of the solve with host checks
    assert counts[1:] == [counts[0] + 1] * 4
