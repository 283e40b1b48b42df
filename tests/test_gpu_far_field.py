"""Merges whose roots' sums use the far-field tables (orders of 2048 and more with 1024 or more
non-deflated poles): block sizes and their edges, and spectra that put blocks on every branch
(uniform, dense at the ends, graded over decades, two clusters, gaps inside blocks), against
the library's tridiagonal solver and by the accuracy ratios of the eigensolver."""
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


def matrix(kind, n):
    g = inputs.SplitMix64(n)
    x = np.arange(n) / n
    e = np.ones(n - 1)
    if kind == "chain":
        return 2.0 + 0.5 * x + 1e-3 * g.uniform(n, -1.0, 1.0), e
    if kind == "hermite":
        return inputs.hermite_tridiag(n)
    if kind == "graded":  # eigenvalues over twelve decades, extended within each
        s = 2.0 ** (-40.0 * x)
        return 2.0 * s, 0.9 * np.sqrt(s[1:] * s[:-1])
    if kind == "bands":  # dimerised chain: two bands with a wide gap
        e[::2] = 0.05
        return 1e-3 * g.uniform(n, -1.0, 1.0) + 0.1 * x, e
    if kind == "step":  # two half chains far apart in energy, weakly coupled everywhere
        return np.where(np.arange(n) % 2 == 0, 0.0, 1e3) + 0.3 * x, e
    raise KeyError(kind)


def check(tdc, d, e):
    n = len(d)
    dt, et = torch.tensor(d, device=DEV), torch.tensor(e, device=DEV)
    lam, Q = tdc.eig(dt, et, check=True)
    T = torch.diag(dt) + torch.diag(et, 1) + torch.diag(et, -1)
    nT = float(lam.abs().max())
    res = float((T @ Q - Q * lam).abs().sum(0).max()) / (n * nT * EPS)
    orth = float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) / (n * EPS)
    assert res <= 50 and orth <= 50
    ref = np.linalg.eigvalsh(np.diag(d) + np.diag(e, 1) + np.diag(e, -1)) if n <= 3000 else None
    if ref is not None:
        assert np.max(np.abs(lam.cpu().numpy() - ref)) <= 10 * n * EPS * nT


@pytest.mark.parametrize("kind", ["chain", "hermite", "graded", "bands", "step"])
@pytest.mark.parametrize("n", [2047, 2048, 2111, 2999])
def test_spectra(tdc, kind, n):
    check(tdc, *matrix(kind, n))


@pytest.mark.parametrize("kind", ["chain", "hermite"])
@pytest.mark.parametrize("n", [4095, 4096, 4161, 8200, 12289])
def test_block_sizes(tdc, kind, n):
    check(tdc, *matrix(kind, n))


@pytest.mark.parametrize("n", [2048, 2300])
def test_band_root(tdc, n):
    """The band solver's top level uses the tables too."""
    AB = inputs.band_sym("laplace", n, 2, seed=3)
    AB[0] += 0.3 * np.arange(n) / n
    lam, Q = tdc.sbevd(torch.tensor(AB, device=DEV), check=True)
    A = torch.diag(torch.tensor(AB[0], device=DEV))
    for r in (1, 2):
        off = torch.diag(torch.tensor(AB[r, :n - r], device=DEV), -r)
        A = A + off + off.t()
    nA = float(lam.abs().max())
    assert float((A @ Q - Q * lam).abs().sum(0).max()) <= 50 * n * nA * EPS
    assert float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) <= 50 * n * EPS
