"""Operator applications captured by the caller after one in FP32: the first FP64
(or float-float) application of a context may be the captured one.  A replay gives
the bits (float-float: the 1e-13 that its varying order leaves) of a direct call."""
import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("precision", ["F64", "FF", "F32C"])
def test_first_application_captured(precision, mode):
    prec = getattr(ibim, "IBIM_" + precision)
    n = 2049
    xs, u, w = inputs.compact_sphere_cloud(n, radius=3.0, seed=8)
    P = ibim.Phys(2.0, 80.0, 0.1257, 0.5, 0)
    side = torch.cuda.Stream()
    x = torch.from_numpy(inputs.random_vector(2 * n, seed=31)).cuda()
    y, z = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    with ibim.Context.from_nodes(xs, u, w, 0.5, stream=side.cuda_stream) as ctx:
        ctx.matvec(P, x, y, precision=ibim.IBIM_F32C)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side, capture_error_mode=mode):
            ctx.matvec(P, x, y, precision=prec)
        x.copy_(torch.from_numpy(inputs.random_vector(2 * n, seed=32)).cuda())
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        ctx.matvec(P, x, z, precision=prec)
        torch.cuda.synchronize()
        if precision == "FF":
            assert float(torch.linalg.norm(y - z)) <= 1e-13 * float(torch.linalg.norm(z))
        else:
            assert torch.equal(y, z)
        del graph
