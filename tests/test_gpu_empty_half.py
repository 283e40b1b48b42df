"""Merges of which one half supports no kept pole: a coupling so weak that only a localised
eigenvector of the other half survives the deflation.  The kept columns are zero in the empty
half's rows, written by FP64 tiles without a single pole; every buffer holds NaN beforehand."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def tdc():
    from paper_2008_01990_gb300 import build, tdc as t
    build.build()
    t.lib()
    return t


def half_empty(n, side):
    """Diagonal on one half of the top split (eigenvectors are unit vectors, the one at the split has
    weight 1 / sqrt 2 in z), a Toeplitz matrix on the other (weights at most sqrt(1 / n2)), coupled by
    b: rho / sqrt 2 > tol >= rho sqrt(1 / n2) for rho = 2 |b| = 1.5 tol, tol = 8 2^-52 max |D|, n2 >= 16."""
    n1 = n // 2
    d, e = np.full(n, 2.0), np.ones(n - 1)
    e[n1 - 1] = 0.75 * 8 * 2.0 ** -52 * 4.0
    lo, hi = (0, n1) if side == "bottom" else (n1, n)
    d[lo:hi] = np.linspace(-3.5, 3.5, hi - lo)
    e[lo:hi - 1] = 0.0
    return d, e


def check(d, e, lam, Q):
    n = len(d)
    assert bool(torch.isfinite(Q).all()) and bool(torch.isfinite(lam).all())
    dd, ee = torch.tensor(d, device=DEV), torch.tensor(e, device=DEV)
    T = torch.diag(dd) + torch.diag(ee, 1) + torch.diag(ee, -1)
    nT = float(torch.linalg.matrix_norm(T, 1))
    assert float((T @ Q - Q * lam).abs().sum(0).max()) <= 50 * n * nT * EPS
    assert float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device=DEV)).abs().sum(0).max()) <= 50 * n * EPS


@pytest.mark.parametrize("side", ["top", "bottom"])
@pytest.mark.parametrize("n", [64, 128, 200, 600, 1500])
def test_one_problem(tdc, n, side):
    d, e = half_empty(n, side)
    o = tdc.default_opts(collect_stats=1)
    ws = torch.full(((tdc.workspace_size(n, o) + 7) // 8,), float("nan"), dtype=torch.float64, device=DEV)
    lam = torch.full((n,), float("nan"), dtype=torch.float64, device=DEV)
    Q = torch.full((n, n), float("nan"), dtype=torch.float64, device=DEV).t()
    tdc.eig(torch.tensor(d, device=DEV), torch.tensor(e, device=DEV), o, ws=ws.view(torch.uint8), lam=lam, Q=Q, check=True)
    assert tdc.get_stats()["sum_K"][0] == 1  # the case that is meant: one pole kept at the top
    check(d, e, lam, Q)


def test_many_problems(tdc):
    """Blocks that walk tiles of several problems: the places of one must not serve another."""
    sizes = np.array([64 + 7 * k for k in range(48)])
    off, offq = np.concatenate([[0], np.cumsum(sizes)]), np.concatenate([[0], np.cumsum(sizes ** 2)])
    d, e = np.zeros(off[-1]), np.zeros(off[-1])
    parts = [half_empty(int(n), "top" if k % 2 else "bottom") for k, n in enumerate(sizes)]
    for k, (a, b) in enumerate(parts):
        d[off[k]:off[k + 1]], e[off[k]:off[k + 1] - 1] = a, b
    ws = torch.full(((tdc.batched_workspace_size(sizes) + 7) // 8,), float("nan"), dtype=torch.float64, device=DEV)
    lam = torch.full((int(off[-1]),), float("nan"), dtype=torch.float64, device=DEV)
    Q = torch.full((int(offq[-1]),), float("nan"), dtype=torch.float64, device=DEV)
    tdc.eig_batched(sizes, torch.tensor(d, device=DEV), torch.tensor(e, device=DEV), off[:-1], offq[:-1], lam, Q,
                    ws=ws.view(torch.uint8), check=True)
    for k, (a, b) in enumerate(parts):
        n = int(sizes[k])
        check(a, b, lam[off[k]:off[k + 1]], Q[offq[k]:offq[k + 1]].view(n, n).t())


@pytest.mark.parametrize("side", ["top", "bottom"])
@pytest.mark.parametrize("n", [2000, 4000, 5001])
def test_empty_half_on_the_split_path(tdc, n, side):
    """The same with more kept poles than the split path's threshold: the full half's eigenvectors at the
    split spread over 200 rows (weights up to sqrt(1 / 201)), the empty half's over all of its n / 2 rows
    (up to sqrt(2 / n)), rho at 0.95 of what would keep the largest of those."""
    n1 = n // 2
    d, e = np.full(n, 2.0), np.ones(n - 1)
    lo, hi, cut = (0, n1, n1 - 200) if side == "bottom" else (n1, n, n1 + 200)
    if side == "bottom":
        d[lo:cut] = np.linspace(-3.5, -0.5, cut - lo)
        e[lo:cut] = 0.0
    else:
        d[cut:hi] = np.linspace(-3.5, -0.5, hi - cut)
        e[cut - 1:hi - 1] = 0.0
    tol = 8 * 2.0 ** -52 * 4.0
    n2 = n - n1 if side == "bottom" else n1
    e[n1 - 1] = 0.5 * 0.95 * tol / np.sqrt(1.0 / (n2 + 1))
    o = tdc.default_opts(collect_stats=1)
    ws = torch.full(((tdc.workspace_size(n, o) + 7) // 8,), float("nan"), dtype=torch.float64, device=DEV)
    lam = torch.full((n,), float("nan"), dtype=torch.float64, device=DEV)
    Q = torch.full((n, n), float("nan"), dtype=torch.float64, device=DEV).t()
    tdc.eig(torch.tensor(d, device=DEV), torch.tensor(e, device=DEV), o, ws=ws.view(torch.uint8), lam=lam, Q=Q, check=True)
    assert 128 <= tdc.get_stats()["sum_K"][0] <= 200
    check(d, e, lam, Q)
