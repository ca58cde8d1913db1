"""Batched solutions against recorded ones: two globules of 24 and 40 atoms, mean
of 32 solves by the symmetric kernel with one target per thread (even shares of
the steps, 48 operations a pair) at 512 sampled unknowns each, with the mean
deviation of one such solve from it (the reverse sums are added in a varying
order; the largest of the 32 was 1.26 times the mean).  A solve whose kernel
rounds alike lies within 1.5 times that deviation."""
import os

import numpy as np
import pytest

from paper_1709_08070_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1709_08070_gb300 import ibim  # noqa: E402

RECORDED = os.path.join(os.path.dirname(__file__), "golden", "batch_solutions.npz")


def test_symmetric_batch_outputs():
    rec = np.load(RECORDED)
    ctxs, phys, outs = [], [], []
    try:
        for m, atoms in enumerate((24, 40)):
            z, r, _ = inputs.globule_atoms(atoms, seed=900 + m)
            q = np.random.default_rng(m).uniform(-0.8, 0.8, len(r))
            ctxs.append(ibim.Context.molecule(z, r, q - q.mean(), probe=1.4, h=0.5, band_eps=1.0))
            phys.append(ibim.Phys(1.0, 80.0, 0.05 * m, 0.5, 0))
            outs.append(torch.empty(2 * ctxs[-1].N, dtype=torch.float64, device="cuda"))
            assert ctxs[-1].N == rec[f"nodes{m}"]
        for v, (_, _, symmetric) in enumerate(ibim.ibim_batch_variants()[0]):
            if not symmetric:
                continue
            ibim.ibim_set_batch_variant(v)
            for _ in range(3):
                ibim.ibim_solve_batch(ctxs, phys, outs, precision=ibim.IBIM_F32C, tol=1e-6, restart=64, maxit=400)
                for m, x in enumerate(outs):
                    at = np.sort(np.random.default_rng(5).choice(x.numel(), 512, replace=False))
                    want = rec[f"p{m}"]
                    far = np.linalg.norm(x.cpu().numpy()[at] - want) / np.linalg.norm(want)
                    assert far <= 1.5 * rec[f"spread{m}"], (v, m, far, float(rec[f"spread{m}"]))
    finally:
        ibim.ibim_set_batch_variant(-1)
        for c in ctxs:
            c.close()
