"""Level-set stages of ibim_build on small and awkward grids against the oracle.

The stage kernel evaluates the second one-sided derivative of an axis only
where a bound asks for it, and works those evaluations off through a queue per
block; the vdW kernel evaluates in FP64 only the atoms an FP32 sweep leaves.
Cases: a grid that is not a multiple of a block, a probe of zero (no flow), a
symmetric pair and a lattice of atoms (kinks on every axis, queues well
filled, many atoms at equal distances) and atoms far from the origin.  About 50 stages of 60 operations round by 2^-53 each
on values of at most 20 A; WENO weights near kinks enlarge that by up to three
orders, so 1e-10 A bounds the difference."""
import numpy as np
import pytest

import oracle
from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402


def _lattice():
    i = np.arange(-1, 2) * 3.0
    return np.stack(np.meshgrid(i, i, i, indexing="ij"), axis=-1).reshape(-1, 3)


CASES = {
    "tiny": (np.zeros((1, 3)), np.array([0.7]), 0.0, 0.5, 1.0),
    "no_flow": (np.array([[0.1, 0.2, 0.3], [2.0, 0.0, 0.0]]), np.array([1.3, 1.7]), 0.0, 0.4, 0.8),
    "pair": (np.array([[-1.5, 0, 0], [1.5, 0, 0]]), np.array([1.5, 1.5]), 1.4, 0.5, 1.5),
    "lattice": (_lattice(), np.full(27, 1.6), 1.4, 0.5, 1.0),
    "far": (inputs.globule_atoms(30)[0] + np.array([400.0, -300.0, 1000.0]), inputs.globule_atoms(30)[1], 1.4, 0.5, 1.0),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_levelset_matches_oracle(name):
    z, r, probe, h, eps = CASES[name]
    ctx = ibim.Context.molecule(z, r, None, probe=probe, h=h, band_eps=eps)
    g, phi_o, _ = oracle.ls_ses(z, r, probe, h, eps)
    lo, n, phi = ctx.levelset()
    assert list(lo) == list(g.lo) and list(n) == list(g.n)
    err = np.max(np.abs(phi - phi_o))
    print("%s: grid %s max |phi - oracle| %.2e" % (name, n, err))
    assert err < 1e-10
    ctx.close()
