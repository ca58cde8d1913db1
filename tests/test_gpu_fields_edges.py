"""Right-hand side and reaction potentials at the edges of their kernels: one
to five charges (one charge per thread block up to three, then four), node
counts around a block, no screening and screening beyond the range of
e^(-kappa rho), against numpy in FP64 with the formulas of the definition.
At most 10^3 terms of 40 operations: 1e-12 of the largest element."""
import math

import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


@pytest.mark.parametrize("kappa", [0.0, 0.1257, 400.0])
@pytest.mark.parametrize("n,nc", [(1, 1), (127, 2), (129, 3), (300, 4), (1000, 5), (257, 300)])
def test_fields_match_definition(n, nc, kappa):
    xs, u, w = inputs.sphere_cloud(n, radius=5.0, seed=n)
    z, q = inputs.kirkwood_charges(n=nc, ball_radius=4.0, seed=nc)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    ctx.set_charges(z, q)
    p = inputs.random_vector(2 * n, seed=4)
    g = torch.empty(2 * n, dtype=torch.float64, device="cuda")
    psi = torch.empty(nc, dtype=torch.float64, device="cuda")
    P = ibim.Phys(2.0, 80.0, kappa, 0.5, 0)
    ctx.rhs(2.0, g)
    gpol = ctx.energy(P, torch.from_numpy(p).cuda(), psi)
    r = xs[:, None, :] - z[None]
    rho = np.linalg.norm(r, axis=2)
    f = 1.0 / (8.0 * math.pi)
    g1 = f * (q / rho).sum(1)
    g2 = -f * (q * (r * u[:, None, :]).sum(2) / rho ** 3).sum(1)
    e = np.exp(-kappa * rho)
    k1 = (1.0 - 40.0 * e * (1 + kappa * rho)) * (r * u[:, None, :]).sum(2) / rho ** 3
    po = ((w * p[:n])[:, None] * k1 + (w * p[n:])[:, None] * (1 - e) / rho).sum(0) / (4 * math.pi)
    got = g.cpu().numpy()
    for a, b in ((got[:n], g1), (got[n:], g2), (psi.cpu().numpy(), po)):
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
    assert abs(gpol - 0.5 * (q * po).sum()) <= 1e-12 * np.abs(q * po).sum()
    ctx.close()


def test_charge_on_a_node_is_infinite_there():
    xs, u, w = inputs.sphere_cloud(64, radius=5.0, seed=1)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    ctx.set_charges(xs[7:8], np.ones(1))
    g = torch.empty(128, dtype=torch.float64, device="cuda")
    ctx.rhs(1.0, g)
    g = g.cpu().numpy()
    assert np.isinf(g[7]) and np.all(np.isfinite(np.delete(g[:64], 7)))
    ctx.close()
