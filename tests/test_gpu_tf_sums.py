"""The three-float running sums of the FP64 near field and of fmm_direct over
many terms whose size rises, falls or jumps along the sources (the constant
the sums run about is raised as they come), of one sign and alternating.

Tolerance per target, as for single pairs: terms accurate to 2^-50, and the
sums lose at most 2^-58 of the largest partial sum per 32 terms (6000 terms:
188 * 2^-58 < 2^-50): |err| <= 2^-49 sum_j |q_j| / r for the potential, 2^-48
sum_j |q_j| / r^2 for each field component."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("signs", ["one", "alternating"])
@pytest.mark.parametrize("order", ["rising", "falling", "mixed"])
def test_many_terms_match_extended_precision(gpu_lib, order, signs):
    fmm = gpu_lib
    rng = np.random.default_rng(5)
    n, nt = 6000, 40
    v = rng.normal(size=(n, 3))
    r = 10.0 ** np.linspace(0.0, -5.0, n)          # distances from the targets' corner: 1 down to 1e-5
    r = {"rising": r, "falling": r[::-1], "mixed": rng.permutation(r)}[order]
    x = np.abs(v / np.linalg.norm(v, axis=1)[:, None]) * r[:, None]
    t = np.sort(rng.choice(n, nt, replace=False))
    x[t] *= 1e-3                                    # the targets, close to the corner
    q = np.ones(n) if signs == "one" else np.where(np.arange(n) % 2, 1.0, -1.0)
    q = q * rng.uniform(0.5, 1.0, n)
    plan = fmm.fmm_plan(torch.from_numpy(x).cuda(), 0, 2, 0.0)
    pot, fld = (a.cpu().numpy()[t] for a in fmm.fmm_eval(plan, torch.from_numpy(q).cuda()))
    dpot, dfld = (a.cpu().numpy() for a in fmm.fmm_direct(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(),
                                                          torch.from_numpy(t).cuda()))
    X, Q = x.astype(np.longdouble), q.astype(np.longdouble)
    d = X[t][:, None, :] - X[None, :, :]
    rr = np.sqrt((d * d).sum(-1))
    w = np.divide(np.longdouble(1), rr, out=np.zeros_like(rr), where=rr > 0)
    phi, mag = (w * Q).sum(1), (w * abs(Q)).sum(1)
    E, magE = ((w ** 3 * Q)[:, :, None] * d).sum(1), (w ** 2 * abs(Q)).sum(1)
    for p, f in ((pot, fld), (dpot, dfld)):
        assert np.all(abs(p - phi) <= 2.0 ** -49 * mag)
        assert np.all(abs(f - E) <= 2.0 ** -48 * magE[:, None])
