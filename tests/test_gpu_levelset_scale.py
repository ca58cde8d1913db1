"""Level set of the same molecule in other units of length: scaling every length by
a power of two is exact in FP64, so phi scales bit for bit, also where the squared
coordinates leave FP32's range."""
import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


@pytest.mark.parametrize("power", [-60, -33, 40, 64, 100])
def test_phi_scales_with_the_unit_of_length(power):
    z, r, _ = inputs.globule_atoms(25, seed=3)
    phis = []
    for s in (1.0, 2.0 ** power):
        with ibim.Context.molecule(s * z, s * r, None, probe=1.5 * s, h=0.5 * s, band_eps=s) as ctx:
            phis.append(ctx.levelset()[2])
    assert np.array_equal(phis[1], 2.0 ** power * phis[0])
