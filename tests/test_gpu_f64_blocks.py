"""FP64 operator at the edges of its 32-node chunks and block pairs.

An item is one unordered pair of blocks of m chunks (m = 1 up to 5,120 nodes);
the sizes cover one node, partly filled chunks, odd and even block counts,
m = 2 and 3 and a last block with fewer chunks, under both tube rules, with
and without screening, and with screening strong enough that e^(-kappa rho)
leaves the normal range.  Every row (the largest cases: 512 rows) against the
oracle: sums of at most 10^4 terms rounded by 2^-53 each with at most 60
operations in front stay below 1e-11 of the largest element."""
import numpy as np
import pytest

import oracle
from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


def _apply(ctx, P, p):
    d = torch.from_numpy(p).cuda()
    y = torch.empty_like(d)
    ctx.matvec(P, d, y, precision=ibim.IBIM_F64)
    first = y.clone()
    ctx.matvec(P, d, y, precision=ibim.IBIM_F64)
    assert torch.equal(first, y)  # fixed summation order: repeats bit for bit
    return y.cpu().numpy()


@pytest.mark.parametrize("kappa,rule", [(0.1257, 0), (0.0, 1), (90.0, 0)])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 97, 1000, 5120, 5153, 10401])
def test_block_edges_match_oracle(n, kappa, rule):
    xs, u, w = inputs.compact_sphere_cloud(n, radius=6.0, seed=n)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    p = inputs.random_vector(2 * n, seed=n + 1)
    y = _apply(ctx, ibim.Phys(1.0, 80.0, kappa, 0.5, rule), p)
    rows = inputs.random_rows(n, 512, seed=3)
    o1, o2 = oracle.matvec_rows(xs, u, w, oracle.Phys(1.0, 80.0, kappa, 0.5, rule), p, rows)
    for got, ref in ((y[:n][rows], o1), (y[n:][rows], o2)):
        assert np.max(np.abs(got - ref)) <= 1e-11 * np.max(np.abs(ref)), np.max(np.abs(got - ref))
    ctx.close()


def test_scattered_order_and_coincident_nodes():
    """A caller order with spread-out chunks, some nodes on top of each other."""
    xs, u, w = inputs.sphere_cloud(700, radius=4.0, seed=9)
    perm = np.random.default_rng(1).permutation(700)
    xs, u, w = xs[perm], u[perm], w[perm]
    xs[40] = xs[39]
    xs[300] = xs[10]
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    p = inputs.random_vector(1400, seed=2)
    y = _apply(ctx, ibim.Phys(2.0, 80.0, 0.1, 0.4, 0), p)
    o1, o2 = oracle.matvec_rows(xs, u, w, oracle.Phys(2.0, 80.0, 0.1, 0.4, 0), p, np.arange(700))
    assert np.max(np.abs(y[:700] - o1)) <= 1e-11 * np.max(np.abs(o1))
    assert np.max(np.abs(y[700:] - o2)) <= 1e-11 * np.max(np.abs(o2))
    ctx.close()
