"""Secular roots of rank-one problems whose poles, weights and rho lie far from one, against
the secular equation solved in 60 digits: the FP32 side of the iteration must not show."""
from decimal import Decimal, getcontext

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def tdc():
    from paper_2008_01990_gb300 import build, tdc as t
    build.build()
    t.lib()
    return t


def true_root(D, z, rho, j, org, start):
    """(tau, sum |t| + 1 / rho, slope) at root j measured from pole org, by safeguarded Newton steps."""
    getcontext().prec = 60
    dl = [Decimal(float(x)) - Decimal(float(D[org])) for x in D]
    zz = [Decimal(float(x)) ** 2 for x in z]
    irho, t = 1 / Decimal(float(rho)), Decimal(float(start))
    lo, hi = dl[j], dl[j + 1] if j + 1 < len(D) else None
    for _ in range(80):
        g = sabs = irho
        gp = Decimal(0)
        for d, w in zip(dl, zz):
            r = 1 / (d - t)
            g += w * r
            sabs += abs(w * r)
            gp += w * r * r
        new = t - g / gp
        if new <= lo:
            new = (t + lo) / 2
        elif hi is not None and new >= hi:
            new = (t + hi) / 2
        if abs(new - t) <= abs(new) * Decimal(10) ** -30:
            return new, sabs, gp
        t = new
    raise AssertionError("no convergence")


# powers of ten of the poles' distances, of z^2 and of rho
SCALES = [(0, 0, 0), (13, 0, 13), (16, 0, 16), (25, 20, 5), (30, 25, 5), (34, 34, 0), (35, 29, 6), (36, 19, 17), (33, 16, 17),
          (-13, 0, -13), (-17, 0, -17), (-25, -38, 13), (-30, -43, 13), (-30, -47, 17), (20, 0, 20), (40, 30, 10)]


@pytest.mark.parametrize("scale", SCALES, ids=lambda s: "D%d_z%d_rho%d" % s)
@pytest.mark.parametrize("K", [3, 33, 40, 300])
def test_roots_at_far_scales(tdc, scale, K):
    """The iteration stops at |g| <= 8 eps (1 / rho + sum |t|).  A term takes 6 roundings (its weight, two
    differences, reciprocal 2, product), the sums K / 32 in a lane, 5 over the warp and 2 at the end: a
    root is within (21 + K / 32) eps sum / slope of the true one, and one rounding of itself."""
    r = np.random.default_rng(K)
    D = (np.sort(r.uniform(0, 1, K)) * 0.9 + np.arange(K)) * 10.0 ** scale[0]
    z = r.uniform(0.2, 1, K) * np.sign(r.standard_normal(K)) * 10.0 ** (scale[1] / 2)
    rho = 10.0 ** scale[2]
    org, tau, _, _ = tdc.rank_one(torch.tensor(D, device=DEV), torch.tensor(z, device=DEV), rho, check=True)
    org, tau = org.cpu().numpy(), tau.cpu().numpy()
    for j in sorted({0, K - 1, *range(0, K, max(1, K // 12))}):
        t, sabs, gp = true_root(D, z, rho, j, int(org[j]), tau[j])
        err = abs(Decimal(float(tau[j])) - t)
        assert err <= Decimal((21 + K / 32) * EPS) * sabs / gp + abs(t) * Decimal(2 * EPS), (j, float(err / abs(t)))


@pytest.mark.parametrize("K", [3, 16, 33, 100, 300])
def test_roots_take_the_last_step(tdc, K):
    """g at an accepted root is known to its own rounding, not only to the test's 8 eps sum, and the step
    that this leaves is taken: errors in units of eps sum / slope are those of g's evaluation.  With 6
    independent roundings of at most one unit a term (0.6 rms each) and up to 5 + K / 32 + 2 in the sums,
    (0.6 sqrt(13 + K / 32)) <= 2.9 units rms for K <= 300, the stopping test alone leaves 8 / sqrt(3) = 4.6."""
    x = []
    for seed in range(12):
        r = np.random.default_rng(100 * K + seed)
        D, z = np.sort(r.uniform(0, 1, K)), r.uniform(0.05, 1, K)
        z /= np.linalg.norm(z)
        org, tau, _, _ = tdc.rank_one(torch.tensor(D, device=DEV), torch.tensor(z, device=DEV), 0.7, check=True)
        org, tau = org.cpu().numpy(), tau.cpu().numpy()
        for j in range(0, K, max(1, K // 10)):
            t, sabs, gp = true_root(D, z, 0.7, j, int(org[j]), tau[j])
            x.append(float((Decimal(float(tau[j])) - t) * gp / sabs / Decimal(EPS)))
    assert np.sqrt(np.mean(np.square(x))) <= 2.9, np.sqrt(np.mean(np.square(x)))
