"""Leaves of 9 to 16 rows (an FP32 solve refined in FP64, or the FP64 QR iteration where that does
not settle), alone and as the leaves of a tree: families that settle at once, that need the 2 x 2
rotations, and that fall back (clusters, grading beyond the FP32 range, decoupled entries)."""
import numpy as np
import pytest
import torch

from paper_2008_01990_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
EPS = np.finfo(float).eps
KINDS = ["uniform", "toeplitz", "wilkinson", "glued", "near", "decoupled", "graded", "steep", "huge", "tiny", "zero"]


@pytest.fixture(scope="module")
def tdc():
    from paper_2008_01990_gb300 import build, tdc as t
    build.build()
    t.lib()
    return t


def matrix(kind, n, seed):
    g = inputs.SplitMix64(1000 * seed + n)
    d, e, x = g.uniform(n, -1.0, 1.0), g.uniform(n - 1, -1.0, 1.0), np.arange(n)
    if kind == "toeplitz":
        return np.full(n, 2.0), np.ones(n - 1)
    if kind == "wilkinson":
        return np.abs(x - (n - 1) / 2.0), np.ones(n - 1)
    if kind == "glued":  # pairs and triples closer than FP32 resolves
        return np.abs(x % 5 - 2.0), np.where(x[1:] % 5 == 0, 1e-9, 1.0)
    if kind == "near":  # one cluster of n eigenvalues
        return 1.0 + 1e-12 * d, 1e-13 * e
    if kind == "decoupled":
        e[::3] = 0.0
        d[1::2] = 0.5
        return d, e
    if kind == "graded":
        s = 2.0 ** (-2.0 * x)
        return s * (2.0 + d), 0.3 * np.sqrt(s[1:] * s[:-1])
    if kind == "steep":
        s = 2.0 ** (-40.0 * x)
        return s * (2.0 + d), 0.3 * np.sqrt(s[1:] * s[:-1])
    if kind == "huge":
        return d * 2.0 ** 400, e * 2.0 ** 400
    if kind == "tiny":
        return d * 2.0 ** -400, e * 2.0 ** -400
    if kind == "zero":
        return np.zeros(n), np.zeros(n - 1)
    return d, e


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [9, 10, 13, 15, 16])
def test_one_leaf(tdc, kind, n):
    """Rounding of the 16-term sums bounds residual and defect by a few n eps; 10 is asked."""
    for seed in range(6):
        d, e = matrix(kind, n, seed)
        lam, Q = tdc.eig(torch.tensor(d, device=DEV), torch.tensor(e, device=DEV), check=True)
        lam, Q = lam.cpu().numpy(), Q.cpu().numpy()
        T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
        nT = max(np.abs(lam).max(), np.abs(T).max())
        assert np.all(np.diff(lam) >= 0)
        assert np.abs(Q.T @ Q - np.eye(n)).sum(0).max() <= 10 * n * EPS
        assert np.abs(T @ Q - Q * lam).sum(0).max() <= 10 * n * EPS * nT


@pytest.mark.parametrize("kind", ["uniform", "glued", "graded", "decoupled"])
@pytest.mark.parametrize("n", [17, 33, 100, 16 * 700])
def test_leaves_of_a_tree(tdc, kind, n):
    """Few leaves and more than the fallback's forms for many (it then takes several a warp)."""
    d, e = matrix(kind, min(n, 400), 7)
    reps = -(-n // len(d))
    d = np.concatenate([d * (1.0 + 0.01 * r) for r in range(reps)])[:n]
    e = np.concatenate([np.append(e, 0.5) for r in range(reps)])[:n - 1]
    lam, Q = tdc.eig(torch.tensor(d, device=DEV), torch.tensor(e, device=DEV), check=True)
    dt, et = torch.tensor(d, device=DEV), torch.tensor(e, device=DEV)
    R = dt[:, None] * Q - Q * lam
    R[1:] += et[:, None] * Q[:-1]
    R[:-1] += et[:, None] * Q[1:]
    nT = float(lam.abs().max())
    assert float(R.abs().sum(0).max()) <= 20 * n * EPS * nT
    assert float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) <= 20 * n * EPS
