"""Switching the float-float kernel between solves: the steps captured for one
kernel are not replayed for the other, so that solves with the one-directional
kernel are equal bit for bit whatever ran before."""
import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


def test_solves_after_a_switch_use_the_chosen_kernel():
    n = 3001
    P = ibim.Phys(2.0, 80.0, 0.1257, 0.5, 0)
    xs, u, w = inputs.compact_sphere_cloud(n, radius=4.0, seed=11)

    def solve(ctx):
        x = torch.empty(2 * n, dtype=torch.float64, device="cuda")
        ctx.solve(P, x, precision=ibim.IBIM_FF, tol=1e-8, certify=0)
        return x

    results = []
    for switched in (False, True):
        with ibim.Context.from_nodes(xs, u, w, 0.5) as ctx:
            ctx.set_charges(np.array([[1.2, 0.0, 0.0], [0.0, -0.8, 0.4]]), np.array([1.0, -0.4]))
            if switched:
                solve(ctx)
            ctx.set_ff_kernel(0)
            results += [solve(ctx) for _ in range(3)]
    assert all(torch.equal(results[0], x) for x in results[1:])
