"""The band tree's levels, whose nodes share their launches: orders around the leaf size (one
leaf, one split, nodes of a level both split and not), every bandwidth class, and spectra that
take the sort's and the deflation's branches, against the library's dense solver."""
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


def dense(AB):
    b, n = AB.shape[0] - 1, AB.shape[1]
    A = np.diag(AB[0])
    for r in range(1, b + 1):
        A += np.diag(AB[r, :n - r], -r) + np.diag(AB[r, :n - r], r)
    return A


def check(tdc, AB):
    """The band solver's own ratios (residual and orthogonality 50), eigenvalues to 10 n eps."""
    n = AB.shape[1]
    A = dense(AB)
    lam, Q = tdc.sbevd(torch.tensor(AB, device=DEV), check=True)
    lam, Q = lam.cpu().numpy(), Q.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    nA = max(np.max(np.abs(ref)), 1e-300)
    assert np.all(np.diff(lam) >= 0)
    assert np.max(np.abs(lam - ref)) <= 10 * n * EPS * nA
    assert np.abs(A @ Q - Q * lam).sum(axis=0).max() <= 50 * n * nA * EPS
    assert np.abs(Q.T @ Q - np.eye(n)).sum(axis=0).max() <= 50 * n * EPS


@pytest.mark.parametrize("n", [2, 127, 128, 129, 255, 257, 259, 515, 1030])
@pytest.mark.parametrize("b", [0, 1, 3, 8])
def test_level_edges(tdc, n, b):
    if b < n:
        check(tdc, inputs.band_sym("uniform", n, b, seed=n + b))


@pytest.mark.parametrize("b,n", [(16, 130), (16, 520), (40, 700), (64, 1100)])
def test_wide_bands(tdc, b, n):
    check(tdc, inputs.band_sym("uniform", n, b, seed=b))


@pytest.mark.parametrize("kind", ["repeat", "decoupled", "zero", "laplace", "graded", "glued"])
@pytest.mark.parametrize("n", [260, 700])
def test_spectra(tdc, kind, n):
    b = 3
    AB = inputs.band_sym(kind if kind in ("laplace", "graded") else "uniform", n, b, seed=7)
    if kind == "repeat":  # the same 20 x 20 block over and over, weakly coupled: many equal poles
        AB = np.tile(AB[:, :20], (1, n // 20 + 1))[:, :n].copy()
        for r in range(1, b + 1):
            AB[r, np.arange(n) % 20 >= 20 - r] *= 1e-14
            AB[r, n - r:] = 0.0
    elif kind == "decoupled":  # no coupling across the splits: every term vanishes
        for r in range(1, b + 1):
            for s in (n // 2, n // 4, n // 2 + (n - n // 2) // 2):
                AB[r, max(0, s - r):s] = 0.0
    elif kind == "zero":
        AB[:] = 0.0
    elif kind == "glued":
        d, e = inputs.glued_wilkinson(n)
        AB = np.zeros((b + 1, n))
        AB[0], AB[1, :n - 1] = d, e
    check(tdc, AB)
