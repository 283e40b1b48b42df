"""Problems of small and large norm: the deflation's tolerance is relative to the matrix, so a
problem times a power of two has the same eigenvectors and its eigenvalues times that power
(bit for bit where both are solved scaled to [1, 2)), and the residual bound of the other
accuracy tests holds at every norm."""
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


def unit(*parts):
    m = np.frexp(max(np.abs(p).max() for p in parts))[1] - 1
    return [np.ldexp(p, -m) for p in parts]


def dev(x):
    return torch.tensor(x, device=DEV)


def ratios(A, lam, Q):
    n, nA = A.shape[0], float(torch.linalg.matrix_norm(A, 1))
    return (float((A @ Q - Q * lam).abs().sum(0).max()) / (n * nA * EPS),
            float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) / (n * EPS))


def dense(AB):
    A = torch.diag(dev(AB[0]))
    for r in range(1, AB.shape[0]):
        low = torch.diag(dev(AB[r, :AB.shape[1] - r].copy()), -r)
        A = A + low + low.t()
    return A


SCALES = [-400, -300, -64, -50, -20, -10, -3, 33, 50, 64, 127, 300, 400]


@pytest.mark.parametrize("k", SCALES)
@pytest.mark.parametrize("n", [5, 16, 300, 2500])
def test_tridiagonal(tdc, n, k):
    d, e = unit(*inputs.uniform_tridiag(n, n))
    lam0, Q0 = tdc.eig(dev(d), dev(e), check=True)
    lam, Q = tdc.eig(dev(np.ldexp(d, k)), dev(np.ldexp(e, k)), check=True)
    assert torch.equal(Q, Q0) and np.array_equal(lam.cpu().numpy(), np.ldexp(lam0.cpu().numpy(), k))
    T = torch.diag(dev(d)) + torch.diag(dev(e), 1) + torch.diag(dev(e), -1)
    res, orth = ratios(T, lam0, Q)
    assert res <= 50 and orth <= 50, (res, orth)


@pytest.mark.parametrize("k", [-64, -20, -3, 50])
def test_band_dense_bidiagonal(tdc, k):
    AB, = unit(inputs.band_sym("uniform", 700, 4, seed=2))
    lam0, Q0 = tdc.sbevd(dev(AB), check=True)
    lam, Q = tdc.sbevd(dev(np.ldexp(AB, k)), check=True)
    assert torch.equal(Q, Q0) and torch.equal(lam, lam0 * 2.0 ** k)
    assert max(ratios(dense(AB), lam0, Q)) <= 50
    A = dev(inputs.dense_sym("uniform", 400, seed=4))
    lam, Z = tdc.syevd(A * 2.0 ** k, check=True)
    assert max(ratios(A, lam * 2.0 ** -k, Z)) <= 50
    d, e = inputs.bidiag_family("uniform", 500, seed=6)
    s, U, VT = tdc.bdsdc(dev(np.ldexp(d, k)), dev(np.ldexp(e, k)), check=True)
    B = torch.diag(dev(d)) + torch.diag(dev(e), 1)
    n, nB = 500, float(torch.linalg.matrix_norm(B, 1))
    assert float((B @ VT.t() - U * (s * 2.0 ** -k)).abs().sum(0).max()) <= 50 * n * nB * EPS


def test_each_problem_of_a_batch_by_itself(tdc):
    n, ks = 200, [0, -30, 40, -3]
    d, e = unit(*inputs.uniform_tridiag(n, 3))
    dd = np.concatenate([np.ldexp(d, k) for k in ks])
    ee = np.concatenate([np.append(np.ldexp(e, k), 0.0) for k in ks])
    off = np.arange(len(ks)) * n
    lam = torch.empty(len(ks) * n, dtype=torch.float64, device=DEV)
    Q = torch.empty(len(ks) * n * n, dtype=torch.float64, device=DEV)
    tdc.eig_batched([n] * len(ks), dev(dd), dev(ee), off, off * n, lam, Q, check=True)
    lam, Q = lam.reshape(-1, n).cpu().numpy(), Q.reshape(len(ks), -1)
    for i, k in enumerate(ks[1:], 1):
        assert torch.equal(Q[i], Q[0]) and np.array_equal(lam[i], np.ldexp(lam[0], k))
