"""GMRES vector kernels at the edges of their blocks and dot-product groups:
vectors shorter than a block, just around one, and of several blocks; restart
lengths below, at and above a group of eight and at the maximum, so that
cycles end inside a group; one system and several of different lengths in one
batched solve.  Solutions against a dense solve of the oracle's operator: the
residual target is 1e-10 and the systems' condition numbers are below 10^3,
so 1e-6 of the solution's norm."""
import numpy as np
import pytest

import oracle
from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402

TAU = 0.5


def _system(n, seed):
    xs, u, w = inputs.compact_sphere_cloud(n, radius=4.0, seed=seed)
    w = w * (4.0 * np.pi * 16.0 / w.sum())  # the sphere's area
    z, q = inputs.kirkwood_charges(n=3, ball_radius=2.0, seed=seed)
    P = oracle.Phys(2.0, 80.0, 0.1257, TAU, 0)
    g = oracle.rhs(xs, u, z, q, 2.0)
    A = np.stack([oracle.matvec(xs, u, w, P, e) for e in np.eye(2 * n)], axis=1)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    ctx.set_charges(z, q)
    return ctx, np.linalg.solve(A, g), g, A


@pytest.mark.parametrize("restart", [7, 8, 9, 17, 128])
@pytest.mark.parametrize("n", [1, 40, 64, 65, 200])
def test_solutions_match_dense_solve(n, restart):
    ctx, x, g, A = _system(n, 5)
    d = torch.empty(2 * n, dtype=torch.float64, device="cuda")
    ctx.solve(ibim.Phys(2.0, 80.0, 0.1257, TAU, 0), d, precision=ibim.IBIM_F64, tol=1e-10, restart=restart, maxit=2000)
    p = d.cpu().numpy()
    assert np.linalg.norm(g - A @ p) <= 2e-10 * np.linalg.norm(g)
    assert np.linalg.norm(p - x) <= 1e-6 * np.linalg.norm(x)
    ctx.close()


def test_batch_of_uneven_lengths():
    sizes = [1, 33, 64, 150, 260]
    systems = [_system(n, 11 + n) for n in sizes]
    P = ibim.Phys(2.0, 80.0, 0.1257, TAU, 0)
    ds = [torch.empty(2 * n, dtype=torch.float64, device="cuda") for n in sizes]
    infos = ibim.ibim_solve_batch([s[0] for s in systems], [P] * len(sizes), ds, tol=1e-6, restart=9, maxit=2000)
    for (ctx, x, g, A), d, info in zip(systems, ds, infos):
        p = d.cpu().numpy()
        assert info["converged"]
        assert np.linalg.norm(g - A @ p) <= 2e-6 * np.linalg.norm(g)
        ctx.close()
