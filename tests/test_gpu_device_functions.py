"""Device functions of the library by themselves (tests/device_functions.cu, compiled against
its headers), against extended precision."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
U = 2.0 ** -53
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2008_01990_gb300 import build
    so = tmp_path_factory.mktemp("device_functions") / "device_functions.so"
    subprocess.run([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "static",
                                                  "-o", str(so), os.path.join(HERE, "device_functions.cu")], check=True)
    return ctypes.CDLL(str(so))


def P(t):
    return ctypes.c_void_p(t.data_ptr())


def dev(x):
    return torch.tensor(np.ascontiguousarray(x, dtype=np.float64), device=DEV)


@pytest.mark.parametrize("log2h", [0, -20, -45])
def test_far_value_and_slope_near_the_points(lib, log2h):
    """The interpolant of a block of half-width h with its far poles at least 4 h from the centre, on
    and around its points.  Value: the sum of 20 weighted values over that of the weights, whose
    rounding is (20 + 6) units of the weights' magnitudes (their ratio is the Lebesgue constant,
    2 / pi log 20 + 1 < 3), so 80 units of Sf, and the truncation 2.4e-18 of it.  Slope: 2^-20 Sf rd3,
    what the root's acceptance takes it to be good to."""
    L, M = np.longdouble, 20
    r = np.random.default_rng(3 - log2h)
    h, yc = 2.0 ** log2h, 0.375 * 2.0 ** log2h
    ang = (2 * np.arange(M) + 1) / (2.0 * M) * np.pi
    y = yc + h * np.cos(ang)
    w = np.where(np.arange(M) & 1, -np.sin(ang), np.sin(ang))
    t = yc + r.choice([-1.0, 1.0], 400) * h * 4 * np.exp(r.uniform(0.01, 8, 400))
    z2 = r.uniform(0, 1, 400)
    term = lambda x: z2.astype(L)[:, None] / (t.astype(L)[:, None] - x.astype(L)[None, :])
    f0, f1 = term(y).sum(0), np.abs(term(y)).sum(0)
    rec = np.concatenate([y, w, f0, f1, np.zeros(M), [0.0, 1 / (3 * h), 0.0, 0.0]])
    off = np.concatenate([[0.0], *[[2.0 ** -k, -2.0 ** -k] for k in range(1, 56)]])
    x = (y[:, None] + h * off[None, :]).ravel()
    x = x[np.abs(x - yc) <= h]
    out = torch.empty(len(x), 4, dtype=torch.float64, device=DEV)
    assert lib.run_far(len(x), P(dev(rec)), P(dev(x)), P(out)) == 0
    out = out.cpu().numpy()
    sf, rd3 = float(f1.max()), 1 / (3 * h)
    assert np.allclose(out[:, 2], sf, rtol=1e-6) and np.allclose(out[:, 3], rd3, rtol=1e-6)
    value, slope = term(x).sum(0), (z2.astype(L)[:, None] / (t.astype(L)[:, None] - x.astype(L)[None, :]) ** 2).sum(0)
    assert np.max(np.abs(out[:, 0] - value)) <= (80 * U + 3e-18) * sf
    assert np.max(np.abs(out[:, 1] - slope)) <= 2.0 ** -20 * sf * rd3
