"""The FP64 rotational M2L at every block size its orders and pair counts take
(Sec. 2.1.3): one warp for a handful of pairs, ragged last warps, runs of
equal targets shorter and longer than a warp, the smallest and largest orders.

Tolerance: the bound this form is held to against the oracle elsewhere, 1e-12
in L2 (here over the locals with every degree scaled to its box, L_k r^k):
the contractions have at most 21 terms and the phases and powers at most 20
products, some 200 unit roundoffs (2e-14) before the conditioning."""
import numpy as np
import pytest
import torch

import oracle
from paper_2002_04894_gb300 import inputs

pytestmark = pytest.mark.gpu

# kind, n, levels, theta: few pairs; many short runs; long runs over several blocks
SIZES = [("uniform", 300, 4, 0.75), ("uniform", 700, 6, 0.7), ("plummer", 4000, 7, 0.6)]


@pytest.mark.parametrize("p", [0, 1, 2, 5, 9, 12, 13, 16, 20])
def test_locals_match_oracle(gpu_lib, p):
    fmm = gpu_lib
    k = np.concatenate([np.full(n + 1, n) for n in range(p + 1)])
    for kind, n, levels, theta in SIZES[:2 if p > 13 else 3]:
        x = inputs.points(kind, n, seed=p)
        q = inputs.charges_uniform(n, seed=p)
        plan = fmm.fmm_plan(torch.from_numpy(x).cuda(), levels, p, theta)
        assert fmm.fmm_plan_stats(plan)["weak_pairs"] > 0
        fmm.fmm_eval(plan, torch.from_numpy(q).cuda())
        T = oracle.Tree(x, levels, p, theta)
        T.eval(q)
        scale = T.tree()["radius"][:, None] ** k
        g, o = fmm.fmm_eval_expansions(plan, "L") * scale, T.expansions("L") * scale
        assert np.linalg.norm(g - o) <= 1e-12 * np.linalg.norm(o), (kind, n)
