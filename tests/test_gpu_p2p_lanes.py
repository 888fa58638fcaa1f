"""Near-field units whose last targets share threads (slices of the sources
per target) and lists cut into segments for few leaves, against the exact sum
(theta = 0: no expansions). Leaf sizes around multiples of 32 and of the 64-
and 128-target tiles, single points, and one leaf.

Tolerances: FP64 form, sums of n terms of relative error <= 16 u each with
cancellation against the sum of magnitudes: n-point L2 error <= 1e-13 at these
sizes (sqrt(n) u growth, u = 1.1e-16). Mixed form: single-precision pairs of
relative error <= 32 u, u = 6e-8, and runs of 64 terms: 2e-6 of the magnitudes
sum's norm."""
import numpy as np
import pytest
import torch

from paper_2002_04894_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,levels", [(1, 0), (2, 1), (31, 0), (33, 0), (65, 0), (95, 0), (129, 0), (141, 0), (63, 3),
                                      (1000, 0), (1000, 3), (130, 1), (5003, 6), (4321, 4), (3000, 7)])
def test_units_of_every_leaf_size(gpu_lib, prec, n, levels):
    fmm = gpu_lib
    x = inputs.points("uniform", n, seed=n)
    q = inputs.charges_uniform(n, seed=n)
    if n > 40:
        x[7] = x[30]  # a coincident pair
    plan = fmm.fmm_plan(torch.from_numpy(x).cuda(), levels, 2, 0.0, prec=prec)
    pot, fld = (t.cpu().numpy() for t in fmm.fmm_eval(plan, torch.from_numpy(q).cuda()))
    d = x[:, None, :] - x[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    w = np.divide(1.0, r, out=np.zeros_like(r), where=r > 0)
    phi, mag = w @ q, w @ np.abs(q)
    E = np.einsum("ij,ijk->ik", w ** 3 * q, d)
    magE = (w ** 2) @ np.abs(q)
    tol = 1e-13 if prec == 0 else 2e-6
    assert np.linalg.norm(pot - phi) <= tol * np.linalg.norm(mag)
    assert np.linalg.norm(fld - E) <= tol * np.linalg.norm(magE)
