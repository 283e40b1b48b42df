"""FP64 merge products around the choice of their tile: one matrix on either side of the order
up to which a level's tiles are few, halves and pole counts next to multiples of the tiles,
and a batch that fills the chip, against the oracle."""
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


def check(d, e, lam, Q):
    """Residual and orthogonality ratios of the eigensolver's tests (50)."""
    n = len(d)
    T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    nT = np.max(np.abs(lam))
    assert np.abs(T @ Q - Q * lam).sum(axis=0).max() <= 50 * n * nT * EPS
    assert np.abs(Q.T @ Q - np.eye(n)).sum(axis=0).max() <= 50 * n * EPS


@pytest.mark.parametrize("mode", ["dense", "auto"])
@pytest.mark.parametrize("n", [63, 65, 127, 129, 257, 511, 1025, 1578, 1580])
def test_single_matrix(tdc, mode, n):
    """1578 is the last order whose top level counts as few tiles (n^2 < 304 x 8192)."""
    d, e = inputs.hermite_tridiag(n)
    o = tdc.default_opts(merge_mode=tdc.MERGE_DENSE if mode == "dense" else tdc.MERGE_AUTO)
    lam, Q = tdc.eig(torch.tensor(d, device=DEV), torch.tensor(e, device=DEV), o, check=True)
    check(d, e, lam.cpu().numpy(), Q.cpu().numpy())


def test_batch_of_wide_merges(tdc):
    """Dense mode, 24 problems of orders 290..330: pole counts above the small tiles' limit."""
    sizes = np.arange(290, 314, dtype=np.int64) + 16
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    offq = np.concatenate([[0], np.cumsum(sizes ** 2)]).astype(np.int64)
    D, E = np.zeros(off[-1]), np.zeros(off[-1])
    for k, n in enumerate(sizes):
        d, e = inputs.hermite_tridiag(int(n))
        D[off[k]:off[k + 1]], E[off[k]:off[k + 1] - 1] = d, e
    lam = torch.empty(int(off[-1]), dtype=torch.float64, device=DEV)
    Q = torch.empty(int(offq[-1]), dtype=torch.float64, device=DEV)
    tdc.eig_batched(sizes, torch.tensor(D, device=DEV), torch.tensor(E, device=DEV), off[:-1], offq[:-1], lam, Q,
                    tdc.default_opts(merge_mode=tdc.MERGE_DENSE), check=True)
    lam, Q = lam.cpu().numpy(), Q.cpu().numpy()
    for k, n in enumerate(sizes):
        check(D[off[k]:off[k + 1]], E[off[k]:off[k + 1] - 1], lam[off[k]:off[k + 1]],
              Q[offq[k]:offq[k + 1]].reshape(n, n).T)
