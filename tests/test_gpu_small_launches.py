"""FP32 operator on small molecules: the untuned choice runs 64-target
tiles up to about 15,000 nodes, the symmetric variants with small
tiles are meant for such sizes, and near chunks run without branches and are
repeated with FP64 decisions only where a tube test is a tie.

Sizes around a chunk, a step, a target tile and the limit; both tube rules, with
screening, without and with strong screening (series and exponential form in
one chunk).  A plane lattice of spacing tau has a tie (rho_P = tau exactly) in
every near chunk.  Against the oracle's rows: FP32 rounds each of about 50
operations by 2^-24 and terms add up with random signs, so 1e-6 of the largest
element (a tube test decided wrongly changes elements by more than 1e-4)."""
import numpy as np
import pytest

import oracle
from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


def _check(ctx, xs, u, w, kappa, tau, rule, variants, seed, rows=256):
    n = len(w)
    p = inputs.random_vector(2 * n, seed=seed)
    d = torch.from_numpy(p).cuda()
    y = torch.empty_like(d)
    pick = inputs.random_rows(n, rows, seed=3)
    o1, o2 = oracle.matvec_rows(xs, u, w, oracle.Phys(1.0, 80.0, kappa, tau, rule), p, pick)
    for v in variants:
        if v is not None:
            ctx.set_f32_variant(v)
        ctx.matvec(ibim.Phys(1.0, 80.0, kappa, tau, rule), d, y, precision=ibim.IBIM_F32C)
        got = y.cpu().numpy()
        for a, b in ((got[:n][pick], o1), (got[n:][pick], o2)):
            assert np.max(np.abs(a - b)) <= 1e-6 * np.max(np.abs(b)), (v, np.max(np.abs(a - b)), np.max(np.abs(b)))


def _variants():
    return [None] + [v for v, info in enumerate(ibim.ibim_f32_variants()) if info[3]]


@pytest.mark.parametrize("n,kappa,rule", [(1, 0.1257, 0), (31, 0.0, 0), (33, 0.1257, 1), (64, 0.4, 0), (65, 3.0, 1),
                                          (127, 0.1257, 0), (129, 0.0, 1), (1000, 0.4, 0), (3001, 0.1257, 0),
                                          (15300, 0.1257, 0), (15500, 0.1257, 0)])
def test_sizes(n, kappa, rule):
    xs, u, w = inputs.compact_sphere_cloud(n, radius=max(1.0, (n / 200.0) ** 0.5), seed=n)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    _check(ctx, xs, u, w, kappa, 0.5, rule, _variants(), seed=n)
    ctx.close()


def test_ties_in_every_near_chunk():
    i = np.arange(24) * 0.5
    xs = np.stack(np.meshgrid(i, i, [0.0, 4.0], indexing="ij"), axis=-1).reshape(-1, 3)
    xs = xs[inputs.bisection_order(xs)]
    u = np.tile([0.0, 0.0, 1.0], (len(xs), 1))
    w = np.random.default_rng(2).uniform(0.01, 0.06, size=len(xs))
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    for rule in (0, 1):
        _check(ctx, xs, u, w, 0.1257, 0.5, rule, [0, 5] + _variants()[1:], seed=6, rows=len(xs))
    ctx.close()
