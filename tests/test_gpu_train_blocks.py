"""Order of the training gradient's sums.  A block of 128 nodes is summed node by
node in FP32, the blocks' sums to float-float and rounded once: with a power of
two as the batch, scaling by it is exact, and the gradient is the rounded FP64
sum of the blocks' own gradients (within one unit of the last place: the
float-float sum is good to 2^-46, so only a near tie can round otherwise).  And a
training call whose launches overlap leaves the parameters that one call per step
leaves."""
import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import warmstart_ref as ws  # noqa: E402
from paper_1709_08070_gb300 import ibim  # noqa: E402

BLOCK = 128


@pytest.fixture(scope="module")
def net():
    n = 20011
    xs, u, w = inputs.compact_sphere_cloud(n, radius=10.0, seed=5)
    ctx = ibim.Context.from_nodes(xs, u, w, 0.5)
    ctx.set_charges(*inputs.kirkwood_charges(n=5, ball_radius=7.0, seed=5))
    P = ibim.Phys(2.0, 80.0, 0.1257, 0.5, 0)
    net = ibim.WarmStartNet(seed=4)
    for k in (1, 2):
        net.add_example(ctx, P, torch.from_numpy(inputs.random_vector(2 * n, seed=20 + k, scale=1e-2)).cuda())
    net.params0 = (0.3 * inputs.random_vector(ws.NPARAMS, seed=14)).astype(np.float32)
    net.set_params(net.params0)
    yield net
    net.close()
    ctx.close()


# 128 blocks, one per CTA; 256 blocks, more than one for most CTAs
@pytest.mark.parametrize("first,count", [(7, 256), (0, 8192), (129, 16384), (0, 32768)])
def test_gradient_is_the_rounded_sum_of_its_blocks(net, first, count):
    net.set_params(net.params0)
    blocks = [net.gradient(first + i, BLOCK)[1].astype(np.float64) for i in range(0, count, BLOCK)]
    exact = np.sum(blocks, axis=0) * (BLOCK / count)
    grad = net.gradient(first, count)[1]
    assert np.all(np.abs(grad - exact) <= np.spacing(np.abs(exact.astype(np.float32))))


@pytest.mark.parametrize("batch", [100, 8192, 30000])
def test_overlapped_steps_equal_single_steps(net, batch):
    runs = []
    for calls, steps in ((1, 6), (6, 1)):
        fresh = ibim.WarmStartNet(seed=4)
        n = 3001
        xs, u, w = inputs.compact_sphere_cloud(n, radius=5.0, seed=6)
        with ibim.Context.from_nodes(xs, u, w, 0.5) as ctx:
            ctx.set_charges(*inputs.kirkwood_charges(n=5, ball_radius=3.5, seed=6))
            fresh.add_example(ctx, ibim.Phys(2.0, 80.0, 0.1257, 0.5, 0),
                              torch.from_numpy(inputs.random_vector(2 * n, seed=23, scale=1e-2)).cuda())
        fresh.set_params(net.params0)
        for _ in range(calls):
            loss = fresh.train(steps, batch_nodes=batch)
        runs.append((loss, fresh.params()))
        fresh.close()
    assert runs[0][0] == runs[1][0] and np.array_equal(runs[0][1], runs[1][1])
