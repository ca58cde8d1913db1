"""Small molecules keep a repeatable FP32 operator: up to 4,608 nodes the
autotuner chooses a one-directional variant, and two applications and two
solves are equal bit for bit, with the small launches (four threads to a target)
among the candidates.  Sizes around a target tile, a source tile and the limit.
Against the oracle's rows to 1e-6 of the largest element (FP32 rounds each of
about 50 operations by 2^-24 and terms add up with random signs)."""
import numpy as np
import pytest

import oracle
from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


@pytest.mark.parametrize("n", [1, 63, 65, 257, 862, 4608])
def test_small_contexts_repeat(n):
    R = max(1.0, (n / 200.0) ** 0.5)
    xs, u, w = inputs.compact_sphere_cloud(n, radius=R, seed=n)
    P = ibim.Phys(2.0, 80.0, 0.1257, 0.5, 0)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    try:
        ctx.set_charges(np.array([[0.3 * R, 0.0, 0.0]]), np.array([1.0]))
        assert ibim.ibim_f32_variants()[ctx.autotune(P)[0]][3] == 0
        p = inputs.random_vector(2 * n, seed=n)
        rows = inputs.random_rows(n, 256, seed=3)
        o = oracle.matvec_rows(xs, u, w, oracle.Phys(2.0, 80.0, 0.1257, 0.5, 0), p, rows)
        d = torch.from_numpy(p).cuda()
        for v in (None, 0):
            if v is not None:
                ctx.set_f32_variant(v)
            ys = []
            for _ in range(2):
                y = torch.empty_like(d)
                ctx.matvec(P, d, y, precision=ibim.IBIM_F32C)
                ys.append(y.cpu().numpy())
            assert np.array_equal(ys[0], ys[1])
            for got, want in ((ys[0][:n][rows], o[0]), (ys[0][n:][rows], o[1])):
                assert np.max(np.abs(got - want)) <= 1e-6 * np.max(np.abs(want))
            xa, xb = torch.empty_like(d), torch.empty_like(d)
            for x in (xa, xb):
                ctx.solve(P, x, precision=ibim.IBIM_F32C, tol=1e-6, restart=64, maxit=400)
            assert torch.equal(xa, xb)
    finally:
        ctx.close()
