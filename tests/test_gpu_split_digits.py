"""The digits of the split products at the edges of their tiles and runs of tiles, and for scales
far from one: whole operands near 2^-480 and 2^480 (a row norm's squares stay in range), with
subnormal and zero entries among them."""
import numpy as np
import pytest
import torch

from oracle import structured as so
from paper_2008_01990_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def tdc():
    from paper_2008_01990_gb300 import build, tdc as t
    build.build()
    t.lib()
    return t


@pytest.mark.parametrize("m,n", [(1, 1), (1, 17), (127, 15), (128, 16), (129, 63), (300, 64), (257, 65), (2000, 129),
                                 (130, 1000)])
@pytest.mark.parametrize("ea,eb", [(0, 0), (-480, 300), (480, -500)])
@pytest.mark.parametrize("slices", [4, 7])
def test_scales(tdc, m, n, ea, eb, slices):
    """Against the product of the operands brought to scale one in FP64: 1e-14 of (largest row
    norm) (column norm) with seven digits, the bound of the products' tests.  With four, a row of
    entries below one and a column scaled to one lose 2^-33 an entry and side, at most n of them
    against a column norm of 2^-1, plus the dropped levels 5 2^-34 a pair at most."""
    A = inputs.SplitMix64(m + n).uniform(m * n, -1.0, 1.0).reshape(m, n)
    t = inputs.SplitMix64(3 * n).uniform(2 * n - 1, -1.0, 1.0)
    A[0, n // 2] = 1.0  # the largest entry, so that no row's scale depends on the draw
    A[m // 2, n // 3] = 0.0 if m > 1 else A[0, n // 3]
    tiny = np.ldexp(A, ea)
    if m > 2:
        tiny[m - 1, n - 1] = 3 * 2.0 ** -1060  # subnormal
    B = so.dense(t, n, 1)
    ref = np.ldexp(tiny, -ea) @ B
    o = tdc.default_opts()
    o.split_slices = slices
    C = tdc.structured_gemm(torch.tensor(np.ascontiguousarray(tiny.T), device=DEV).t(),
                            torch.tensor(np.ldexp(t, eb), device=DEV), tdc.TOEPLITZ, tdc.MERGE_SPLIT, opts=o, check=True)
    got = np.ldexp(C.cpu().numpy(), -ea - eb)
    scale = np.linalg.norm(A, axis=1).max() * np.linalg.norm(B, axis=0)[None, :]
    tol = 1e-14 if slices == 7 else 1e-14 + n * 2.0 ** -28
    assert np.max(np.abs(got - ref) / scale) <= tol
