"""Leaves of 33 to 64 rows, and few leaves of 17 to 32 (two warps a leaf), in a workspace that holds
NaN beforehand: the same bits every time, and the residual and orthogonality bounds of the others."""
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


@pytest.mark.parametrize("n,leaf", [(1, 64), (2, 64), (33, 64), (64, 64), (300, 32), (900, 32), (1000, 64), (4000, 64)])
@pytest.mark.parametrize("family", ["uniform", "toeplitz"])
def test_two_warp_leaves_repeat_bitwise(tdc, n, leaf, family):
    d, e = inputs.uniform_tridiag(n, n) if family == "uniform" else inputs.toeplitz_tridiag(n)
    d, e = torch.tensor(d, device=DEV), torch.tensor(e, device=DEV)
    o = tdc.default_opts(leaf=leaf)
    ws = torch.empty((tdc.workspace_size(n, o) + 7) // 8, dtype=torch.float64, device=DEV)
    ref = None
    for _ in range(20):
        ws.fill_(float("nan"))
        lam = torch.full((n,), float("nan"), dtype=torch.float64, device=DEV)
        Q = torch.full((n, n), float("nan"), dtype=torch.float64, device=DEV).t()
        tdc.eig(d, e, o, ws=ws.view(torch.uint8), lam=lam, Q=Q, check=True)
        if ref is None:
            ref = lam, Q
            T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
            nT = float(torch.linalg.matrix_norm(T, 1))
            assert float((T @ Q - Q * lam).abs().sum(0).max()) <= 50 * n * nT * EPS
            assert float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) <= 50 * n * EPS
        else:
            assert torch.equal(lam, ref[0]) and torch.equal(Q, ref[1])
