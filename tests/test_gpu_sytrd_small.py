"""Reductions of at most one column a block, in a workspace that holds NaN beforehand: an
exchanged value that is read before it is written would show, and every repetition gives the
same bits."""
import ctypes

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


@pytest.mark.parametrize("first", range(3, 161, 16))
def test_small_orders_repeat_bitwise(tdc, first):
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    for n in range(first, min(first + 16, 161)):
        A = torch.tensor(inputs.dense_sym("uniform", n, seed=n), device=DEV)
        nb = ctypes.c_size_t(0)
        assert tdc.lib().tdc_sytrd_workspace_size(n, ctypes.byref(nb)) == 0
        ws = torch.empty((nb.value + 7) // 8, dtype=torch.float64, device=DEV)
        ref = None
        for _ in range(200 if n in (3, 4, 5, 31, 32, 33, 100, 151, 152, 153) else 20):
            ws.fill_(float("nan"))
            R = A.t().contiguous().t()
            d, e, tau = (torch.full((n,), float("nan"), dtype=torch.float64, device=DEV) for _ in range(3))
            st = tdc.lib().tdc_sytrd(n, P(R), n, P(d), P(e), P(tau), P(ws), ws.numel() * 8, None,
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
            assert st == 0
            got = [d, e[:n - 1], tau[:n - 1], R]
            if ref is None:
                assert tdc.sync_status() == 0
                ref = got
                # Q^T A Q = T to the reduction's backward error, n eps ||A||_F entry-wise, twice over
                Q = torch.eye(n, dtype=torch.float64, device=DEV).t().contiguous().t()
                tdc.ormtr(R, tau[:n - 1], Q, check=True)
                T = torch.diag(d) + torch.diag(e[:n - 1], 1) + torch.diag(e[:n - 1], -1)
                nA = float(torch.linalg.norm(A))
                assert float((Q.t() @ A @ Q - T).abs().max()) <= 2 * n * EPS * nA, n
            else:
                for x, y in zip(ref, got):
                    assert torch.equal(x, y), n
        assert tdc.sync_status() == 0
