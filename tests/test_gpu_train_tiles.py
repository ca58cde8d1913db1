"""Training gradient at the edges of its 64-node tiles and of a CTA's share of
them: one node, around a tile, a tile per CTA on every SM and more, and ranges
that do not start at a tile.  Loss and gradient against the FP64 numpy network;
FP32 sums of at most 2 10^4 terms with a relative error of 2^-24 each stay below
1e-5 of the gradient's norm.  The sums run in a fixed order, so two calls agree
bit for bit."""
import numpy as np
import pytest

from oracle import warmstart_ref as ws
from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


@pytest.fixture(scope="module")
def net():
    n = 20011
    xs, u, w = inputs.compact_sphere_cloud(n, radius=10.0, seed=3)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    z, q = inputs.kirkwood_charges(n=5, ball_radius=7.0, seed=3)
    ctx.set_charges(z, q)
    P = ibim.Phys(2.0, 80.0, 0.1257, 0.5, 0)
    net = ibim.WarmStartNet(seed=2)
    params = (0.3 * inputs.random_vector(ws.NPARAMS, seed=12)).astype(np.float32)
    net.set_params(params)
    p = inputs.random_vector(2 * n, seed=13, scale=1e-2)
    net.add_example(ctx, P, torch.from_numpy(p).cuda())
    feat, scales = net.features(ctx, P)
    target, weight = ws.targets(p, w, scales, 2.0, 80.0)
    yield net, ws.bf16_round(params), feat.astype(np.float64), np.asarray(target), np.asarray(weight)
    net.close()
    ctx.close()


@pytest.mark.parametrize("first,count", [(0, 1), (5, 63), (64, 64), (1, 65), (0, 9728), (3, 9729), (0, 20011)])
def test_gradient_matches_reference(net, first, count):
    n, params, feat, target, weight = net
    loss, grad = n.gradient(first, count)
    again = n.gradient(first, count)
    assert loss == again[0] and np.array_equal(grad, again[1])
    s = slice(first, first + count)
    loss_o, grad_o = ws.loss_and_grad(params, feat[s], target[s], weight[s])
    assert loss == pytest.approx(loss_o, rel=1e-5)
    assert np.linalg.norm(grad - grad_o) <= 1e-5 * np.linalg.norm(grad_o)
