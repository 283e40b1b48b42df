"""Secular roots (tdc_rank_one) around the window of 32 poles and on the spectra that take the
solver's branches: weights over 14 decades (roots 1e-28 of the interval from their pole),
clustered and graded poles, widely scaled problems.  Each root is judged by the secular
function itself in extended precision."""
import numpy as np
import pytest
import torch

from paper_2008_01990_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def tdc():
    from paper_2008_01990_gb300 import build, tdc as t
    build.build()
    t.lib()
    return t


def problem(kind, K, seed):
    g = inputs.SplitMix64(seed)
    D = np.sort(g.uniform(K, -1.0, 1.0)) + 1e-9 * np.arange(K)
    z = g.uniform(K, 0.1, 1.0)
    rho = 0.7
    if kind == "tiny":  # weights from 1 down to 1e-14, in random order
        z = z * 10.0 ** -(14.0 * g.uniform01(K))
    elif kind == "cluster":  # groups of poles a few thousand eps apart
        D = np.floor(np.arange(K) / 7.0) + 1e-12 * (np.arange(K) % 7)
    elif kind == "graded":
        D = 2.0 ** (-40.0 * np.arange(K)[::-1] / K)
        z = z * D
    elif kind == "one":  # one weight carries everything
        z = 1e-8 * z
        z[K // 2] = 1.0
    elif kind == "huge":  # outside the range of the FP32 estimate
        D, rho = D * 2.0 ** 150, rho * 2.0 ** 150
    elif kind == "small":
        D, rho = D * 2.0 ** -150, rho * 2.0 ** -150
    return D, z / np.linalg.norm(z), rho


@pytest.mark.parametrize("kind", ["uniform", "tiny", "cluster", "graded", "one", "huge", "small"])
@pytest.mark.parametrize("K", [1, 2, 16, 31, 32, 33, 47, 48, 63, 64, 65, 127, 500])
def test_roots_satisfy_the_secular_equation(tdc, kind, K):
    D, z, rho = problem(kind, K, 1000 + K)
    org, tau, zhat, s = tdc.rank_one(torch.tensor(D, device=DEV), torch.tensor(z, device=DEV), rho, check=True)
    org, tau = org.cpu().numpy(), tau.cpu().numpy()
    x = np.longdouble
    zz = x(z) ** 2
    for j in range(K):
        o = int(org[j])
        assert o == j or (o == j + 1 and j < K - 1)
        width = D[j + 1] - D[j] if j < K - 1 else rho * float(np.sum(zz)) * (1 + K * EPS)
        assert (0 < tau[j] <= width) if o == j else (-width <= tau[j] < 0)
        dl = (x(D) - x(D[o])) - x(tau[j])
        t = zz / dl
        g, slope = 1 / x(rho) + t.sum(), (t / dl).sum()
        # accepted at |g| <= 8 eps (1/rho + sum |t|) as computed (sums of K terms in FP64 by
        # lanes: as much again), or by a step below the rounding of tau
        assert abs(g) <= 16 * EPS * (1 / x(rho) + np.abs(t).sum()) + 4 * EPS * abs(tau[j]) * slope
