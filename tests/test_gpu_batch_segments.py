"""Batched symmetric kernels: steps cut into large segments and small ones
from a counter, one and two targets per thread.

Sizes at the edges of a warp, a source step and a target tile (512 and 1,024),
a single molecule with fewer steps than CTAs, and molecules with more steps
than CTAs, so that segments begin inside rows and end inside other molecules.
Checked by the residual of each batched solution under the FP64 operator: the
solver's tolerance of 1e-6 plus the FP32 operator's relative error (1e-6 of
the largest element, with |A x| a few times |b|), so 1e-5."""
import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


@pytest.mark.parametrize("sizes", [(1,), (513,), (31, 1023, 1025, 2049), (20000, 1, 7001, 512, 256)])
def test_segments(sizes):
    P = ibim.Phys(1.0, 80.0, 0.1257, 0.5, 0)
    ctxs = []
    try:
        for k, n in enumerate(sizes):
            R = max(1.0, (n / 200.0) ** 0.5)
            xs, u, w = inputs.compact_sphere_cloud(n, radius=R, seed=n + k)
            ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
            ctx.set_charges(np.array([[0.3 * R, 0.0, 0.0], [0.0, -0.2 * R, 0.1 * R]]), np.array([1.0, -0.4]))
            ctxs.append(ctx)
        for v, (_, _, symmetric) in enumerate(ibim.ibim_batch_variants()[0]):
            if not symmetric:
                continue
            ibim.ibim_set_batch_variant(v)
            outs = [torch.empty(2 * c.N, dtype=torch.float64, device="cuda") for c in ctxs]
            infos = ibim.ibim_solve_batch(ctxs, [P] * len(ctxs), outs, precision=ibim.IBIM_F32C, tol=1e-6, restart=64,
                                          maxit=400)
            assert ibim.ibim_batch_variants()[1] == v
            for ctx, x, info in zip(ctxs, outs, infos):
                b = torch.empty_like(x)
                ctx.rhs(P.eps_in, b)
                y = torch.empty_like(x)
                ctx.matvec(P, x, y, precision=ibim.IBIM_F64)
                res = float(torch.linalg.norm(y - b) / torch.linalg.norm(b))
                assert info["converged"] and res <= 1e-5, (v, ctx.N, res)
    finally:
        ibim.ibim_set_batch_variant(-1)
        for c in ctxs:
            c.close()
