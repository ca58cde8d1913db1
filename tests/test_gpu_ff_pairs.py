"""Float-float operator in packed pairs of nodes: sizes around a half chunk, a
chunk and a target tile, both kernels and tube rules, without and with strong
screening, a tube wider than the cloud's chunks, and a lattice of spacing tau
with a tie (rho_P = tau exactly) in every near chunk.  Against the oracle to
the 1e-10 of max |y| per element that the operator is held to (float-float
rounds at 2^-47 or so; a tube test decided wrongly changes elements by more
than 1e-4)."""
import numpy as np
import pytest

import oracle
from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


def _check(xs, u, w, kappa, tau, rule):
    n = len(w)
    p = inputs.random_vector(2 * n, seed=n)
    o = oracle.matvec(xs, u, w, oracle.Phys(2.0, 80.0, kappa, tau, rule), p)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    try:
        for symmetric in (1, 0):
            ctx.set_ff_kernel(symmetric)
            y = ctx.matvec_host(ibim.Phys(2.0, 80.0, kappa, tau, rule), p, precision=ibim.IBIM_FF)
            for b in (slice(0, n), slice(n, 2 * n)):
                assert np.max(np.abs(y[b] - o[b])) <= 1e-10 * np.max(np.abs(o[b])), (symmetric, b)
    finally:
        ctx.close()


@pytest.mark.parametrize("n,kappa,tau,rule", [(15, 0.1257, 0.5, 0), (16, 0.0, 0.5, 1), (17, 3.0, 0.5, 0),
                                              (31, 0.1257, 0.1, 1), (32, 0.0, 0.5, 0), (127, 0.1257, 2.0, 0),
                                              (129, 1.0, 0.5, 1), (1025, 0.1257, 0.5, 0), (2000, 0.4, 3.0, 0)])
def test_sizes(n, kappa, tau, rule):
    xs, u, w = inputs.compact_sphere_cloud(n, radius=max(1.0, (n / 30.0) ** 0.5), seed=n)
    _check(xs, u, w, kappa, tau, rule)


@pytest.mark.parametrize("rule", [0, 1])
def test_ties(rule):
    i = np.arange(16) * 0.5
    xs = np.stack(np.meshgrid(i, i, [0.0, 4.0], indexing="ij"), axis=-1).reshape(-1, 3)
    xs = xs[inputs.bisection_order(xs)]
    u = np.tile([0.0, 0.0, 1.0], (len(xs), 1))
    _check(xs, u, np.full(len(xs), 0.02), 0.1257, 0.5, rule)
