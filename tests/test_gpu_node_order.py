"""Node order of built geometries: every range of the recursive bisection is
split across the longest side of its bounding box at the documented place, with
no node of the left part beyond one of the right.  Sizes below and above the
one where halves are ordered by several threads; two builds agree exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim, inputs  # noqa: E402


def _check(xs, lo, hi):
    n = hi - lo
    if n <= 32:
        return
    part = xs[lo:hi]
    axis = int(np.argmax(part.max(axis=0) - part.min(axis=0)))
    unit = 1024 if n >= 2048 else (256 if n >= 512 else 32)
    k = unit * max(1, int(np.floor(n / (2.0 * unit) + 0.5)))
    assert part[:k, axis].max() <= part[k:, axis].min()
    _check(xs, lo, lo + k)
    _check(xs, lo + k, hi)


@pytest.mark.parametrize("radius", [1.0, 4.0, 9.0, 20.0])
def test_sphere(radius):
    ctx = ibim.Context.sphere(radius, centre=(0.1, 0.2, -0.3), h=0.5)
    xs = ctx.nodes()["xs"]
    again = ibim.Context.sphere(radius, centre=(0.1, 0.2, -0.3), h=0.5)
    assert np.array_equal(xs, again.nodes()["xs"])
    _check(xs, 0, len(xs))
    ctx.close()
    again.close()


def test_globule():
    z, r, q = inputs.globule_atoms(300)
    ctx = ibim.Context.molecule(z, r, q, probe=1.4, h=0.5, band_eps=1.0)
    xs = ctx.nodes()["xs"]
    assert len(xs) > 32768
    _check(xs, 0, len(xs))
    ctx.close()
