"""The power-of-two scales of the split products' operands (A's largest row norm, the column
bounds of Toeplitz / Hankel and Cauchy-like operands) at the edges of their kernels: a bound
that misses a row, a generator or a node lets digits overflow, which the products show."""
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


@pytest.mark.parametrize("m", [1, 7, 8, 9, 2431, 2432, 2433, 2447, 4863, 4864, 4865])
@pytest.mark.parametrize("n", [1, 31, 129])
def test_row_scale_edges(tdc, m, n):
    """The largest row (2^20 times the others) sits at the first, a middle and the last row:
    error within 1e-14 of (largest row norm) (column norm), the bound of the products' tests
    with A's rows at one scale."""
    t = inputs.SplitMix64(n).uniform(2 * n - 1, -1.0, 1.0)
    B = so.dense(t, n, 1)
    base = inputs.SplitMix64(m + n).uniform(m * n, -1.0, 1.0).reshape(m, n)
    for row in {0, m // 2, m - 1}:
        A = base.copy()
        A[row] *= 2.0 ** 20
        At = torch.tensor(np.ascontiguousarray(A.T), device=DEV).t()
        C = tdc.structured_gemm(At, torch.tensor(t, device=DEV), tdc.TOEPLITZ, tdc.MERGE_SPLIT, check=True)
        scale = np.linalg.norm(A, axis=1).max() * np.linalg.norm(B, axis=0)[None, :]
        assert np.max(np.abs(C.cpu().numpy() - A @ B) / np.maximum(scale, 1e-300)) <= 1e-14


@pytest.mark.parametrize("kind", [1, 2])
@pytest.mark.parametrize("n", [1, 2, 511, 512, 513, 1025])
def test_window_scale_edges(tdc, kind, n):
    """One generator 2^30 times the others, at the ends, next to the middle and in between:
    the columns that hold it take its scale, the others keep theirs."""
    base = inputs.SplitMix64(n + kind).uniform(2 * n - 1, -1.0, 1.0)
    A = inputs.SplitMix64(5 * n).uniform(40 * n, -1.0, 1.0).reshape(40, n)
    At = torch.tensor(np.ascontiguousarray(A.T), device=DEV).t()
    for at in sorted({0, n // 3, max(n - 2, 0), n - 1, min(n, 2 * n - 2), (3 * n) // 2 % (2 * n - 1), 2 * n - 2}):
        t = base.copy()
        t[at] = 2.0 ** 30
        B = so.dense(t, n, kind)
        C = tdc.structured_gemm(At, torch.tensor(t, device=DEV), kind, tdc.MERGE_SPLIT, check=True).cpu().numpy()
        scale = np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(B, axis=0)[None, :]
        assert np.max(np.abs(C - A @ B) / scale) <= 1e-14


@pytest.mark.parametrize("n", [33, 500])
@pytest.mark.parametrize("e", [-1005, 990])
def test_cauchy_scale_of_extreme_nodes(tdc, n, e):
    """Nodes and weights times 2^e: the same B, from differences outside the range in which
    the norms take the hardware reciprocal (spacings near 2^-1015) or near its end."""
    d, w, u, v = inputs.example1_cauchy(n)
    A = inputs.SplitMix64(n).uniform(64 * n, -1.0, 1.0).reshape(64, n)
    At = torch.tensor(np.ascontiguousarray(A.T), device=DEV).t()
    out = []
    for x in (0, e):
        g = [torch.tensor(np.ldexp(q, x), device=DEV) for q in (d, w, u)]
        out.append(tdc.cauchy_like_gemm(At, g[0], g[1], g[2], torch.tensor(v, device=DEV), tdc.MERGE_SPLIT,
                                        check=True).cpu().numpy())
    B = u[:, None] * v[None, :] / (d[:, None] - w[None, :])
    scale = np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(B, axis=0)[None, :]
    assert np.max(np.abs(out[1] - out[0]) / scale) <= 1e-14
