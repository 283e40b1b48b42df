"""FP64 merge products of levels of many merges (32768 rows and more): 64-row and 32-row tiles in
one level, halves on either side of multiples of both, against the residual and orthogonality
bounds of the eigensolver's tests (50)."""
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


@pytest.mark.parametrize("mode", ["dense", "auto"])
@pytest.mark.parametrize("orders", [(127, 128, 129, 130), (254, 255, 256, 257, 258), (191, 193, 320, 322, 386),
                                    (704, 705, 767, 770)])
def test_orders(tdc, mode, orders):
    sizes = np.array([orders[k % len(orders)] for k in range(-(-33000 // min(orders)))], dtype=np.int64)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    offq = np.concatenate([[0], np.cumsum(sizes ** 2)]).astype(np.int64)
    D, E = np.zeros(off[-1]), np.zeros(off[-1])
    for k, n in enumerate(sizes):
        d, e = inputs.hermite_tridiag(int(n))
        D[off[k]:off[k + 1]], E[off[k]:off[k + 1] - 1] = d + 0.01 * k * np.arange(n) / n, e
    lam = torch.empty(int(off[-1]), dtype=torch.float64, device=DEV)
    Q = torch.empty(int(offq[-1]), dtype=torch.float64, device=DEV)
    o = tdc.default_opts(merge_mode=tdc.MERGE_DENSE if mode == "dense" else tdc.MERGE_AUTO)
    dt, et = torch.tensor(D, device=DEV), torch.tensor(E, device=DEV)
    tdc.eig_batched(sizes, dt, et, off[:-1], offq[:-1], lam, Q, o, check=True)
    for k in list(range(2 * len(orders))) + list(range(len(sizes) - len(orders), len(sizes))):
        n = int(sizes[k])
        l = lam[off[k]:off[k + 1]]
        V = Q[offq[k]:offq[k + 1]].reshape(n, n).t()
        T = torch.diag(dt[off[k]:off[k + 1]]) + torch.diag(et[off[k]:off[k + 1] - 1], 1)
        T = T + torch.triu(T, 1).t()
        assert float((T @ V - V * l).abs().sum(0).max()) <= 50 * n * EPS * float(l.abs().max())
        assert float((V.t() @ V - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) <= 50 * n * EPS
