"""The autotuner's cache over its limit of 4,608 nodes for repeatable variants,
which lies inside a size bucket: a choice made above it is not handed to a
smaller context, which has to repeat bit for bit, nor one made below to a larger
context, for which the symmetric variants were timed."""
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402

P = ibim.Phys(2.0, 80.0, 0.1257, 0.5, 0)
SMALL, LARGE = 4300, 8000


def _context(n):
    return ibim.Context.from_nodes(*inputs.compact_sphere_cloud(n, radius=(n / 200.0) ** 0.5, seed=n), 0.5)


def _tuned(n):
    with _context(n) as ctx:
        v = ctx.autotune(P)[0]
    return v, ibim.ibim_f32_variants()[v][3] != 0


def _applications(ctx, count):
    x = torch.from_numpy(inputs.random_vector(2 * ctx.N, seed=9)).cuda()
    ys = [torch.empty_like(x) for _ in range(count)]
    for y in ys:
        ctx.matvec(P, x, y, precision=ibim.IBIM_F32C)
    return ys


def test_choice_above_the_limit_stays_above():
    if not _tuned(LARGE)[1]:
        pytest.skip("the measured choice at %d nodes is one-directional here" % LARGE)
    with _context(SMALL) as ctx:
        first, *others = _applications(ctx, 6)
        assert all(torch.equal(first, y) for y in others)


def test_choice_below_the_limit_stays_below():
    if not _tuned(LARGE)[1]:
        pytest.skip("the measured choice at %d nodes is one-directional here" % LARGE)
    small, symmetric = _tuned(SMALL)
    assert not symmetric
    with _context(LARGE) as ctx:
        kept, = _applications(ctx, 1)
        ctx.set_f32_variant(small)
        assert not torch.equal(kept, _applications(ctx, 1)[0])
