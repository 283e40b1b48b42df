"""Band solves in a workspace that holds NaN beforehand, repeated: the same bits every time.
Orders whose upper nodes have more rows than the deflation's block has threads, and bands of
which all, half or few of a node's poles deflate by their weight (localised eigenvectors on
both sides of the splits, on one side, on none)."""
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


def band(kind, n, b):
    AB = inputs.band_sym("uniform" if kind == "localised" else "laplace", n, b, seed=n)
    if kind == "half":
        AB[:, :n // 2] = inputs.band_sym("uniform", n, b, seed=n)[:, :n // 2]
    return AB


@pytest.mark.parametrize("kind", ["localised", "half", "extended"])
@pytest.mark.parametrize("n,b", [(300, 4), (1100, 3), (2600, 2)])
def test_band_solves_repeat_bitwise(tdc, kind, n, b):
    P = lambda t: ctypes.c_void_p(t.data_ptr())
    AB = band(kind, n, b)
    ABc = torch.tensor(np.ascontiguousarray(AB.T), device=DEV)
    nb = ctypes.c_size_t(0)
    assert tdc.lib().tdc_sbevd_workspace_size(n, b, None, ctypes.byref(nb)) == 0
    ws = torch.empty((nb.value + 7) // 8, dtype=torch.float64, device=DEV)
    ref = None
    for _ in range(12):
        ws.fill_(float("nan"))
        lam = torch.full((n,), float("nan"), dtype=torch.float64, device=DEV)
        Q = torch.full((n, n), float("nan"), dtype=torch.float64, device=DEV)
        assert tdc.lib().tdc_sbevd(n, b, P(ABc), b + 1, P(lam), P(Q), n, P(ws), ws.numel() * 8, None,
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        assert tdc.sync_status() == 0
        if ref is None:
            ref = lam, Q
            # the band solver's own ratios: residual and orthogonality 50
            A = torch.diag(torch.tensor(AB[0], device=DEV))
            for r in range(1, b + 1):
                low = torch.diag(torch.tensor(AB[r, :n - r].copy(), device=DEV), -r)
                A = A + low + low.t()
            V, nA = Q.t(), float(lam.abs().max())
            assert float((A @ V - V * lam).abs().sum(0).max()) <= 50 * n * nA * EPS
            assert float((V.t() @ V - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) <= 50 * n * EPS
        else:
            assert torch.equal(lam, ref[0]) and torch.equal(Q, ref[1])
