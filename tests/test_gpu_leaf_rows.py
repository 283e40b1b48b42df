"""Leaf eigensolves on their own (problems of at most the leaf size are one leaf, no merge):
every variant of the leaf kernels by leaf size and number of leaves, on the inputs that take
its branches (zero, tiny, huge-ratio and equal entries), against the dense library solver."""
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


def leaf_problem(kind, n, seed):
    d, e = inputs.uniform_tridiag(n, seed)
    if kind == 1:  # already diagonal
        e = 0.0 * e
    elif kind == 2:  # closed form, shift at the centre
        d, e = 0.0 * d, 0.0 * e + 1.0
    elif kind == 3:  # decoupled pieces
        e[::3] = 0.0
    elif kind == 4:  # entries down to 2^-1000: squares underflow
        s = 2.0 ** np.floor(-1000.0 * np.arange(n) / max(n - 1, 1))
        d, e = d * s, e * s[1:]
    elif kind == 5:  # off-diagonals around the negligibility threshold
        e = e * 2.0 ** -(48.0 + 8.0 * inputs.SplitMix64(seed).uniform01(n - 1))
    elif kind == 6:  # equal diagonal, weak coupling
        d, e = 0.0 * d + 1.0, e * 1e-9
    elif kind == 7:  # all zero
        d, e = 0.0 * d, 0.0 * e
    return d, e


@pytest.mark.parametrize("leaf,lo", [(8, 1), (16, 9), (32, 17)])
@pytest.mark.parametrize("count", [1, 65, 1217, 2433, 4001])
def test_leaves_against_library(tdc, leaf, lo, count):
    sizes = inputs.SplitMix64(leaf + count).integers(count, lo, leaf)
    sizes[0] = leaf  # the variant goes by the largest leaf
    probs = [leaf_problem(k % 8, int(n), 17 * k + leaf) for k, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    offq = np.concatenate([[0], np.cumsum(sizes * sizes)]).astype(np.int64)
    D, E = np.zeros(off[-1]), np.zeros(off[-1])
    for k, (d, e) in enumerate(probs):
        D[off[k]:off[k + 1]] = d
        E[off[k]:off[k + 1] - 1] = e
    lam = torch.empty(int(off[-1]), dtype=torch.float64, device=DEV)
    Q = torch.empty(int(offq[-1]), dtype=torch.float64, device=DEV)
    tdc.eig_batched(sizes, torch.tensor(D, device=DEV), torch.tensor(E, device=DEV), off[:-1], offq[:-1], lam, Q,
                    tdc.default_opts(leaf=leaf), check=True)
    lam, Q = lam.cpu().numpy(), Q.cpu().numpy()
    for k, (d, e) in enumerate(probs):
        n = int(sizes[k])
        T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
        v, U = lam[off[k]:off[k + 1]], Q[offq[k]:offq[k + 1]].reshape(n, n).T
        # QR iteration: backward error of a few eps per rotation passing an entry (about 2 n)
        tol = 10 * n * EPS
        nrm = max(np.max(np.abs(np.linalg.eigvalsh(T))), 1e-300)
        assert np.all(np.diff(v) >= 0)
        assert np.max(np.abs(v - np.linalg.eigvalsh(T))) <= tol * nrm
        assert np.max(np.abs(T @ U - U * v)) <= tol * nrm
        assert np.max(np.abs(U.T @ U - np.eye(n))) <= tol
