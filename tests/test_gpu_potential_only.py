"""Evaluations without the field run near-field kernels of their own: the FP64
form's and the mixed form's two tile sizes, with and without segmented lists,
sliced targets, both result types, and batches in which some systems have a field
array and others none.

theta = 0 (the exact sum, no expansions). Tolerances as for the evaluations with the
field (test_gpu_p2p_lanes.py): 1e-13 and 2e-6 of the magnitudes sum's norm; float32
results are rounded once more, by 2^-24 of the value."""
import numpy as np
import pytest
import torch

from paper_2002_04894_gb300 import inputs

pytestmark = pytest.mark.gpu

# whole tiles and left-over targets of 32-, 64- and 128-target units; one leaf, a few (segments), many
SIZES = [(1, 0), (33, 0), (141, 0), (63, 3), (130, 1), (1000, 3), (5003, 6), (3000, 7)]


def exact(x, q):
    d = x[:, None, :] - x[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    w = np.divide(1.0, r, out=np.zeros_like(r), where=r > 0)
    return w @ q, w @ np.abs(q)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,levels", SIZES)
def test_potential_without_the_field(gpu_lib, n, levels, prec, dtype):
    fmm = gpu_lib
    x = torch.from_numpy(inputs.points("uniform", n, seed=n)).to(dtype)
    q = torch.from_numpy(inputs.charges_uniform(n, seed=n)).to(dtype)
    if n > 40:
        x[7] = x[30]  # a coincident pair
    plan = fmm.fmm_plan(x.cuda(), levels, 2, 0.0, prec=prec)
    pot, fld = fmm.fmm_eval(plan, q.cuda(), want_fields=False)
    assert fld is None and pot.dtype == dtype
    phi, mag = exact(x.double().numpy(), q.double().numpy())
    tol = (1e-13 if prec == 0 else 2e-6) + (2.0 ** -24 if dtype == torch.float32 else 0.0)
    assert np.linalg.norm(pot.double().cpu().numpy() - phi) <= tol * np.linalg.norm(mag)


@pytest.mark.parametrize("with_field", [(True, False, True, False), (False, False, False, False), (False, True, False, False)])
def test_batch_where_some_systems_have_no_field(gpu_lib, with_field):
    """Each system's results are those of its own evaluation with what it asks for,
    and nothing is written for a system without a field array."""
    fmm = gpu_lib
    plans, qs, pots, flds, refs = [], [], [], [], []
    for i, (n, levels) in enumerate([(900, 3), (5003, 6), (3000, 7), (40, 0)]):
        x = torch.from_numpy(inputs.points("plummer", n, seed=i).astype(np.float32))
        q = torch.from_numpy(inputs.charges_uniform(n, seed=i).astype(np.float32))
        plans.append(fmm.fmm_plan(x.cuda(), levels, 6, 0.0, prec=fmm.FMM_PREC_MIXED))
        qs.append(q.cuda())
        pots.append(torch.full((n,), float("nan"), device="cuda"))
        flds.append(torch.full((n, 3), float("nan"), device="cuda") if with_field[i] else None)
        refs.append(fmm.fmm_eval(plans[-1], qs[-1], want_fields=True))
    torch.cuda.synchronize()
    batch = fmm.fmm_batch_create(plans, qs, pots, flds)
    assert fmm.fmm_batch_info(batch)["fused"]
    fmm.fmm_batch_launch(batch)
    torch.cuda.synchronize()
    for (p, f), pot, fld in zip(refs, pots, flds):
        assert float((pot - p).norm() / p.norm()) <= 1e-6
        if fld is not None:
            assert float((fld - f).norm() / f.norm()) <= 1e-6
