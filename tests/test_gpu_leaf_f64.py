"""FP64 P2M and L2P at the sizes where their tiles end: leaves of 1 to 300
points (warps of 32, blocks of 128), orders whose coefficient count ends a
batch of eight or leaves a remainder, the smallest and largest orders.

Tolerance: the bound this form is held to against the oracle elsewhere, 1e-12
in L2 (multipoles with every degree scaled to its box, M_n / r^n): recurrences
of at most 20 steps and sums of at most 300 terms, under 500 unit roundoffs
(6e-14)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2002_04894_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [1, 31, 32, 33, 128, 129, 300])
@pytest.mark.parametrize("p", [0, 1, 3, 6, 10, 14, 20])
def test_multipoles_and_far_field_match_oracle(gpu_lib, p, leaf):
    fmm = gpu_lib
    levels = 5
    n = leaf << levels
    x = inputs.points("uniform", n, seed=leaf)
    q = inputs.charges_uniform(n, seed=p)
    plan = fmm.fmm_plan(torch.from_numpy(x).cuda(), levels, p, 0.75)
    assert fmm.fmm_plan_stats(plan)["weak_pairs"] > 0
    pot, fld = fmm.fmm_eval(plan, torch.from_numpy(q).cuda())
    T = oracle.Tree(x, levels, p, 0.75)
    op, oE = T.eval(q)
    first = (1 << levels) - 1
    r = np.maximum(T.tree()["radius"][first:, None], 1e-300)
    k = np.concatenate([np.full(m + 1, m) for m in range(p + 1)])
    scale = np.where(r > 1e-200, r, 1.0) ** -k
    g, o = fmm.fmm_eval_expansions(plan, "M")[first:] * scale, T.expansions("M")[first:] * scale
    assert np.linalg.norm(g - o) <= 1e-12 * np.linalg.norm(o)
    assert np.linalg.norm(pot.cpu().numpy() - op) <= 1e-12 * np.linalg.norm(op)
    assert np.linalg.norm(fld.cpu().numpy() - oE) <= 1e-12 * np.linalg.norm(oE)
