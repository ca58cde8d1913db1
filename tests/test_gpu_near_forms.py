"""The branch-free near chunks (small launches, symmetric variants) against the
branching ones (the other one-directional variants).  On one source tile all
one-directional variants form the same sums: equal bit for bit, the tube tests
decided alike.  Two patches 40.3 Angstrom apart, every pair of opposite nodes within
a thousandth of the tangent-plane cylinder of radius 0.37, under tube rule 1: a
pair decided otherwise changes its row by 1e-5 of the largest element or more; the
symmetric variants round their sums differently by 1e-6 at most.  (Those that reduce
across the warp take near pairs by a scalar form, whose rho^2 rounds otherwise: not
compared on the patches.)"""
import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


def _patches(n, tau):
    rng = np.random.default_rng(4)
    xs, u = np.zeros((n, 3)), np.zeros((n, 3))
    half = n // 2
    xs[:, 1:] = np.tile(rng.uniform(-1.0, 1.0, (half, 2)), (2, 1))
    xs[half:, 0] = 40.3
    angle, off = rng.uniform(0.0, 2.0 * np.pi, half), tau * (1.0 + rng.uniform(-1e-3, 1e-3, half))
    xs[half:, 1] += off * np.cos(angle)
    xs[half:, 2] += off * np.sin(angle)
    u[:half, 0], u[half:, 0] = -1.0, 1.0
    turn = np.linalg.qr(rng.standard_normal((3, 3)))[0]
    return xs @ turn.T, u @ turn.T, rng.uniform(0.01, 0.11, n)


@pytest.mark.parametrize("case", ["patches", "cloud", "ragged"])
@pytest.mark.parametrize("rule", [0, 1])
def test_near_forms_agree(case, rule):
    tau = 0.37
    if case == "patches":
        xs, u, w = _patches(256, tau)
    else:
        n = 256 if case == "cloud" else 97
        xs, u, w = inputs.compact_sphere_cloud(n, radius=1.3, seed=n)
    n = len(w)
    P = ibim.Phys(2.0, 80.0, 0.1257, tau, rule)
    x = torch.from_numpy(inputs.random_vector(2 * n, seed=6)).cuda()
    ys = []
    with ibim.Context.from_nodes(xs, u, w, 0.5) as ctx:
        kinds = [v[3] for v in ibim.ibim_f32_variants()]
        for v in range(len(kinds)):
            ctx.set_f32_variant(v)
            y = torch.empty_like(x)
            ctx.matvec(P, x, y, precision=ibim.IBIM_F32C)
            ys.append(y)
    plain = [v for v, k in enumerate(kinds) if k == 0]
    assert all(torch.equal(ys[plain[0]], ys[v]) for v in plain[1:])
    for kind, y in zip(kinds, ys):
        if kind == 1 and case == "patches":
            continue
        for part in (slice(0, n), slice(n, 2 * n)):
            assert float((y[part] - ys[plain[0]][part]).abs().max()) <= 1e-6 * float(ys[plain[0]][part].abs().max())
