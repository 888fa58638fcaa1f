"""The register-resident single-precision M2L (orders 1..12, Sec. 2.1.3
rotation form) against the FP64 M2L on the same points.

Tolerance, from the operation count: five chained contractions of at most
p + 1 terms in single precision (unit roundoff 2^-24), and the float P2M
before them (sums of depth <= 16): the local expansions, every degree scaled to
its box (L_k r^k), differ by at most (5 (p + 1) + 16) 2^-24 of their norm."""
import numpy as np
import pytest
import torch

from paper_2002_04894_gb300 import inputs

pytestmark = pytest.mark.gpu

# kind, n, levels, theta: few pairs (part of one warp's 32), many short target runs, long lists, a ragged tail
SIZES = [("uniform", 300, 4, 0.7), ("uniform", 700, 5, 0.7), ("plummer", 6000, 9, 0.5), ("gmm", 20000, 8, 0.6)]


def scaled_locals(fmm, plan, p):
    L = fmm.fmm_eval_expansions(plan, "L")
    k = np.concatenate([np.full(n + 1, n) for n in range(p + 1)])
    return L * fmm.fmm_plan_tree(plan)["radius"][:, None] ** k


@pytest.mark.parametrize("p", range(1, 13))
def test_locals_match_fp64(gpu_lib, p):
    fmm = gpu_lib
    for kind, n, levels, theta in SIZES:
        x = torch.from_numpy(inputs.points(kind, n, seed=p)).cuda()
        q = torch.from_numpy(inputs.charges_uniform(n, seed=p)).cuda()
        got = []
        for prec in (fmm.FMM_PREC_FP64, fmm.FMM_PREC_MIXED):
            plan = fmm.fmm_plan(x, levels, p, theta, prec=prec)
            fmm.fmm_eval(plan, q)
            fmm.fmm_eval_check(plan)
            assert fmm.fmm_plan_stats(plan)["weak_pairs"] > 0
            got.append(scaled_locals(fmm, plan, p))
        err = np.linalg.norm(got[1] - got[0]) / np.linalg.norm(got[0])
        assert err <= (5 * (p + 1) + 16) * 2.0 ** -24, (kind, n, err)


@pytest.mark.parametrize("p", [1, 5, 9, 11, 12])
def test_batch_equals_alone(gpu_lib, p):
    """Systems of different pair counts (none, part of a warp, ragged) in one batch."""
    fmm = gpu_lib
    plans, qs, pots, alone = [], [], [], []
    for i, (kind, n, levels) in enumerate([("uniform", 40, 1), ("uniform", 700, 5), ("plummer", 9000, 7), ("gmm", 3000, 6)]):
        x = torch.from_numpy(inputs.points(kind, n, seed=i).astype(np.float32)).cuda()
        q = torch.from_numpy(inputs.charges_uniform(n, seed=i).astype(np.float32)).cuda()
        plans.append(fmm.fmm_plan(x, levels, p, 0.6, prec=fmm.FMM_PREC_MIXED))
        alone.append(fmm.fmm_eval(plans[-1], q)[0])
        qs.append(q)
        pots.append(torch.zeros(n, device="cuda"))
    torch.cuda.synchronize()
    batch = fmm.fmm_batch_create(plans, qs, pots)
    assert fmm.fmm_batch_info(batch)["fused"]
    fmm.fmm_batch_launch(batch)
    for plan, a, b in zip(plans, alone, pots):
        fmm.fmm_eval_check(plan)
        # the same sums in another order of the double atomics: a float ulp or two (as the other batch tests hold)
        assert float((a - b).norm() / a.norm()) <= 1e-6


@pytest.mark.parametrize("p", [2, 4])
def test_overflow_stays_with_its_target(gpu_lib, p):
    """A charge so large that its M2L into the boxes near it overflows in single
    precision, in a long thin box whose far end it reaches with finite values: the
    targets there, which share warps with the overflowing ones, are not touched.
    Tolerance against the FP64 form: as above for the expansions, and as much again
    for the near field's runs and L2P."""
    fmm = gpu_lib
    n = 3000
    xn = inputs.points("uniform", n, seed=p) * np.array([0.03, 3e-4, 3e-4])
    xn[0] = [0.0, 1.5e-4, 1.5e-4]
    qn = inputs.charges_uniform(n, seed=p) * 1e30
    qn[0] = 1e36
    x, q = torch.from_numpy(xn).cuda(), torch.from_numpy(qn).cuda()
    pot = []
    for prec in (fmm.FMM_PREC_FP64, fmm.FMM_PREC_MIXED):
        plan = fmm.fmm_plan(x, 9, p, 0.5, prec=prec)
        pot.append(fmm.fmm_eval(plan, q)[0].cpu().numpy())
    far = xn[:, 0] > 0.0125                    # potentials of 3.3e37 to 8e37
    assert far.sum() > 1000
    assert not np.isfinite(fmm.fmm_eval_expansions(plan, "L")).all()   # (the overflow does happen)
    err = np.abs(pot[1][far] - pot[0][far]).max() / np.abs(pot[0][far]).max()
    assert err <= 2 * (5 * (p + 1) + 16) * 2.0 ** -24, err


@pytest.mark.parametrize("p", [8, 12])
def test_constant_term_of_one_pair(gpu_lib, p):
    """What the axial sum loses in a local expansion's constant term: two clusters of
    positive charges, one weak pair each way. Half the difference of the two boxes'
    relative errors, each less its source's monopole's, is free of the roundings both
    share (the distance's reciprocal) and of P2M's. The sum's terms fall with the
    degree, and one chain from the smallest up is to lose less than two chains added
    at the end (as orders 14 and 16 sum). Tolerance, from an emulation of the same
    20,000 pairs' roundings (root mean square in 2^-24): 0.73 with two chains, 0.91
    with one from the largest down, 0.44 from the smallest up."""
    fmm = gpu_lib
    rng = np.random.default_rng(p)
    half = []
    for _ in range(200):
        d = rng.normal(size=3)
        d *= 2.0 / rng.uniform(0.3, 0.45) / np.linalg.norm(d)
        xn = rng.uniform(-1, 1, (80, 3)) / np.sqrt(3.0)
        xn[40:] += d
        x, q = torch.from_numpy(xn).cuda(), torch.from_numpy(rng.uniform(0, 1, 80)).cuda()
        got = {}
        for prec in (fmm.FMM_PREC_FP64, fmm.FMM_PREC_MIXED):
            plan = fmm.fmm_plan(x, 1, p, 0.5, prec=prec, tight=True)
            fmm.fmm_eval(plan, q)
            assert fmm.fmm_plan_stats(plan)["weak_pairs"] == 2
            got[prec] = [fmm.fmm_eval_expansions(plan, w)[1:, 0].real for w in "LM"]
        (l0, m0), (l1, m1) = got[fmm.FMM_PREC_FP64], got[fmm.FMM_PREC_MIXED]
        e = (l1 / l0 - 1) - (m1 / m0 - 1)[::-1]
        half.append((e[0] - e[1]) / 2)
    rms = np.sqrt(np.mean(np.square(half)))
    assert rms <= 0.73 * 2.0 ** -24, rms * 2.0 ** 24
