"""The reduction's last columns in the SMs' shared memory (one exchange a column), at the
orders where its layout changes: below, at and above one column a block, the largest order it
takes, and panels of the blocked reduction before it."""
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


def check_reduction(tdc, A):
    """Q^T A Q = T and Q^T Q = I to the reduction's backward error (O(n) rounding errors per
    entry and reflector: n eps ||A||_F entry-wise, with the factor 10 of the oracle's pins over 5)."""
    n = A.shape[0]
    At = torch.tensor(A, device=DEV)
    d, e, tau, R = tdc.sytrd(At, check=True)
    Q = torch.eye(n, dtype=torch.float64, device=DEV).t().contiguous().t()
    tdc.ormtr(R, tau, Q, check=True)
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    nA = float(torch.linalg.norm(At))
    assert float((Q.t() @ At @ Q - T).abs().max()) <= 2 * n * EPS * nA
    assert float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device=DEV)).abs().max()) <= 2 * n * EPS
    return d, e


@pytest.mark.parametrize("n", [3, 4, 5, 31, 151, 152, 153, 154, 155, 304, 305, 513, 1823, 1824, 1825, 1953])
def test_reduction_at_layout_edges(tdc, n):
    check_reduction(tdc, inputs.dense_sym("uniform", n, seed=n))


@pytest.mark.parametrize("name", ["zerocol", "tridiag", "lowrank", "cluster"])
@pytest.mark.parametrize("n", [160, 700])
def test_reduction_of_degenerate_columns(tdc, name, n):
    """Trivial reflectors (tau = 0) and columns at rounding level."""
    check_reduction(tdc, inputs.dense_sym(name, n, seed=n))


def test_same_result_twice_and_after_other_sizes(tdc):
    """The blocks' meeting counter starts from zero in every call, and no exchanged vector of
    an earlier call in the same workspace is ever taken for this call's."""
    A, B = (torch.tensor(inputs.dense_sym("uniform", n, seed=n), device=DEV) for n in (401, 640))
    ref = [x.clone() for x in tdc.sytrd(A, check=True)]
    for _ in range(3):
        tdc.sytrd(B, check=True)
        for x, y in zip(ref, tdc.sytrd(A, check=True)):
            assert torch.equal(x, y)


def test_wait_that_runs_out_is_reported(tdc):
    A = torch.tensor(inputs.dense_sym("uniform", 900, seed=9), device=DEV)
    with pytest.raises(tdc.TdcError) as err:
        tdc.sytrd(A, tdc.default_opts(spin_budget=1), check=True)
    assert err.value.status == tdc.TDC_ETIMEOUT
    check_reduction(tdc, inputs.dense_sym("uniform", 300, seed=300))
