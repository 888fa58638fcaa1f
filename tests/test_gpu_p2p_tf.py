"""The FP64 form's near field (three-float arithmetic, FP64 for the pairs it
cannot hold) against the exact sum in extended precision, theta = 0.

Tolerance per target: a pair's terms are accurate to 2^-52 relative (FP64
pairs: a few ulp, < 2^-50), the sums add less, and the result is rounded once:
|err| <= 2^-49 sum_j |q_j| / r for the potential, 2^-48 sum_j |q_j| / r^2 for each
field component."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def cloud(kind, n, rng):
    x = rng.random((n, 3))
    q = rng.uniform(-1.0, 1.0, n)
    if kind == "close":          # distances from 1e-1 down to 1e-15 around a few points
        x = x[rng.integers(0, 5, n)] + 10.0 ** rng.uniform(-15, -1, (n, 1)) * rng.normal(size=(n, 3))
        x[3] = x[9]
    elif kind == "centre":       # fine bits: clusters at the root cell's centre and at the origin
        x = (x - 0.5) * 10.0 ** rng.uniform(-12, 0, (n, 1))
        x[0], x[1] = (-0.5, -0.5, -0.5), (0.5, 0.5, 0.5)
    elif kind == "offset":
        x = x + 1.0e6
    elif kind == "huge":
        x = x * 1e120
    elif kind == "tiny":
        x, q = x * 1e-120, q * 1.6e-19
    elif kind == "charges":      # magnitudes from 1 down to 1e-40, zeros
        q = q * 10.0 ** rng.uniform(-40, 0, n)
        q[::7] = 0.0
    elif kind == "plane":
        x[:, 2] = 0.25
    elif kind == "line":
        x[:, 1:] = 0.0
    return x, q


@pytest.mark.parametrize("levels", [0, 3])
@pytest.mark.parametrize("kind", ["uniform", "close", "centre", "offset", "huge", "tiny", "charges", "plane", "line"])
def test_matches_extended_precision(gpu_lib, kind, levels):
    fmm = gpu_lib
    x, q = cloud(kind, 333, np.random.default_rng(17))
    plan = fmm.fmm_plan(torch.from_numpy(x).cuda(), levels, 2, 0.0)
    pot, fld = (t.cpu().numpy() for t in fmm.fmm_eval(plan, torch.from_numpy(q).cuda()))
    X, Q = x.astype(np.longdouble), q.astype(np.longdouble)
    d = X[:, None, :] - X[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    w = np.divide(np.longdouble(1), r, out=np.zeros_like(r), where=r > 0)
    phi, mag = (w * Q).sum(1), (w * abs(Q)).sum(1)
    E, magE = ((w ** 3 * Q)[:, :, None] * d).sum(1), (w ** 2 * abs(Q)).sum(1)
    assert np.all(abs(pot - phi) <= 2.0 ** -49 * mag)
    assert np.all(abs(fld - E) <= 2.0 ** -48 * magE[:, None])


def test_non_finite_charge_reaches_every_target(gpu_lib):
    fmm = gpu_lib
    x, q = cloud("uniform", 100, np.random.default_rng(3))
    for bad in (np.inf, np.nan):
        q[41] = bad
        plan = fmm.fmm_plan(torch.from_numpy(x).cuda(), 2, 2, 0.0)
        pot = fmm.fmm_eval(plan, torch.from_numpy(q).cuda())[0].cpu().numpy()
        assert not np.isfinite(pot).any()


@pytest.mark.parametrize("nt", [1, 33, 129, 333])
@pytest.mark.parametrize("kind", ["uniform", "close", "centre", "offset", "huge", "tiny", "charges", "plane"])
def test_direct_matches_extended_precision(gpu_lib, kind, nt):
    fmm = gpu_lib
    x, q = cloud(kind, 333, np.random.default_rng(23))
    t = np.arange(nt)[::-1].copy()
    pot, fld = (v.cpu().numpy() for v in fmm.fmm_direct(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(),
                                                        torch.from_numpy(t).cuda()))
    X, Q = x.astype(np.longdouble), q.astype(np.longdouble)
    d = X[t][:, None, :] - X[None, :, :]
    r = np.sqrt((d * d).sum(-1))
    w = np.divide(np.longdouble(1), r, out=np.zeros_like(r), where=r > 0)
    phi, mag = (w * Q).sum(1), (w * abs(Q)).sum(1)
    E, magE = ((w ** 3 * Q)[:, :, None] * d).sum(1), (w ** 2 * abs(Q)).sum(1)
    assert np.all(abs(pot - phi) <= 2.0 ** -49 * mag)
    assert np.all(abs(fld - E) <= 2.0 ** -48 * magE[:, None])


def test_direct_slabs_and_bad_indices(gpu_lib):
    """More sources than one slab of records (2^20), float32, targets out of range and next to the slab's end."""
    fmm = gpu_lib
    n = (1 << 20) + 1001
    rng = np.random.default_rng(5)
    x, q = rng.random((n, 3)).astype(np.float32), rng.uniform(-1, 1, n).astype(np.float32)
    t = np.array([0, -1, (1 << 20) - 1, 1 << 20, n, n - 1])
    pot, fld = (v.cpu().numpy() for v in fmm.fmm_direct(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(),
                                                        torch.from_numpy(t).cuda()))
    assert np.isnan(pot[[1, 4]]).all() and np.isnan(fld[[1, 4]]).all()
    X, Q = x.astype(np.float64), q.astype(np.float64)
    for k in (0, 2, 3, 5):
        d = X[t[k]] - X
        r = np.sqrt((d * d).sum(1))
        w = np.divide(1.0, r, out=np.zeros_like(r), where=r > 0)
        # float32 results: one rounding (2^-24) beside the reference's own 1e-12
        assert abs(pot[k] - (w * Q).sum()) <= 2.0 ** -23 * abs((w * Q).sum()) + 1e-12 * (w * abs(Q)).sum()
        E = ((w ** 3 * Q)[:, None] * d).sum(0)
        assert np.all(abs(fld[k] - E) <= 2.0 ** -23 * abs(E) + 1e-12 * (w ** 2 * abs(Q)).sum())


def test_direct_long_sums_of_pairs_left_to_fp64(gpu_lib):
    """A far outlier (every pair of the cluster is then left to FP64) and many targets
    (few segments: a thread adds some 30,000 terms of one sign). Tolerance: the terms'
    own roundings in FP64, at most 4 2^-53 of 1/r and 11 2^-53 of d/r^3, and 2 2^-53
    for compensated sums and the result."""
    fmm = gpu_lib
    n = 100_000
    rng = np.random.default_rng(29)
    x, q = rng.random((n, 3)), rng.uniform(0.5, 1.0, n)
    x[0] = 1e8, 0.0, 0.0
    pot, fld = (v.cpu().numpy() for v in fmm.fmm_direct(torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda(),
                                                        torch.arange(n, device="cuda")))
    X, Q = x.astype(np.longdouble), q.astype(np.longdouble)
    for t in range(1, n, n // 12):
        d = X[t] - X
        r = np.sqrt((d * d).sum(1))
        w = np.divide(np.longdouble(1), r, out=np.zeros_like(r), where=r > 0)
        assert abs(pot[t] - (w * Q).sum()) <= 6 * 2.0 ** -53 * (w * Q).sum()
        assert np.all(abs(fld[t] - ((w ** 3 * Q)[:, None] * d).sum(0)) <= 13 * 2.0 ** -53 * (w ** 2 * Q).sum())
