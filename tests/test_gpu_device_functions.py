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


def wide(r, n, lo, hi):
    """Mantissas over [1, 2) at binary exponents lo .. hi, both signs."""
    return r.uniform(1, 2, n) * 2.0 ** r.integers(lo, hi + 1, n) * r.choice([-1.0, 1.0], n)


@pytest.mark.parametrize("lo,hi", [(-4, 4), (-470, 470), (-530, 505)])
def test_reciprocals_and_reflectors(lib, lo, hi):
    """Units u = 2^-53 of relative error.  rsqrt_cubic: its argument's product and last sum, 2 (the
    refinement leaves 2^-60); rsqrt_nr: two steps of four roundings, 4; rcp_nr: 2.  reflector: the norm
    t2 1 (half in its root), 1 / beta 2.5, beta 4.5, alpha - beta 5.5, its reciprocal 7.5, tau 9.  Outside
    [2^-960, 2^960] of t2 the library's root and divisions, as good; orders where even alpha^2 + s leaves
    FP64 are the callers' (their input is scaled)."""
    L, r, n = np.longdouble, np.random.default_rng(hi), 40000
    a = wide(r, n, lo, hi)
    with np.errstate(over="ignore"):
        b = np.abs(wide(r, n, -40, 40)) * a * a
    b = np.clip(b, 2.0 ** -1021, 2.0 ** 1022)
    keep = (np.abs(a) > 2.0 ** -505) if lo < -505 else np.ones(n, bool)
    out = torch.empty(n, 6, dtype=torch.float64, device=DEV)
    assert lib.run_scalars(n, P(dev(a)), P(dev(b)), P(out)) == 0
    out = out.cpu().numpy()
    al, bl = a.astype(L), b.astype(L)
    nrm = np.sqrt(al * al + bl)
    beta = np.where(al < 0, nrm, -nrm)
    for q, ref, units in [(0, 1 / np.sqrt(np.abs(al)), 2), (1, 1 / np.sqrt(np.abs(al)), 4), (5, 1 / al, 2),
                          (3, beta, 5), (4, 1 / (al - beta), 8), (2, (beta - al) / beta, 9)]:
        err = (np.abs(out[:, q] - ref) / np.abs(ref))[keep]
        assert np.max(err) <= units * U, (q, float(np.max(err) / U))


def test_rotations(lib):
    """w: its square 1.5 (half of it in the root), 1 / w 2.75, w 4.25; c and s 3.75 units; beyond the
    range hypot (2 ulp, up to 4 units) and divisions, 5.  Weights down to 2^-530 and one of the two zero."""
    L, r, n = np.longdouble, np.random.default_rng(8), 40000
    a, b = wide(r, n, -530, 500), wide(r, n, -530, 500)
    near = r.random(n) < 0.5
    b[near] = (a * wide(r, n, -60, 60))[near]
    b[::50] = 0.0
    out = torch.empty(n, 3, dtype=torch.float64, device=DEV)
    assert lib.run_rotation(n, P(dev(a)), P(dev(b)), P(out)) == 0
    out = out.cpu().numpy()
    w = np.sqrt(a.astype(L) ** 2 + b.astype(L) ** 2)
    for q, ref in [(0, w), (1, a / w), (2, -b / w)]:
        big = np.abs(ref) > 2.0 ** -1000
        err = np.abs(out[:, q] - ref)[big] / np.abs(ref)[big]
        assert np.max(err) <= 6 * U, (q, float(np.max(err) / U))


def test_joint_warp_sums(lib):
    """The sums of two and three values at once: exact on integers, in every lane, and otherwise
    five additions' worth of rounding."""
    r, n = np.random.default_rng(9), 300
    for v in (r.integers(-1000, 1000, (n, 3, 32)).astype(float), wide(r, n * 96, -30, 30).reshape(n, 3, 32)):
        out = torch.empty(n, 6, 32, dtype=torch.float64, device=DEV)
        assert lib.run_sums(n, P(dev(v)), P(out)) == 0
        out = out.cpu().numpy()
        ref, mag = v.astype(np.longdouble).sum(2), np.abs(v).sum(2)
        for q, row in enumerate([0, 1, 0, 1, 2, 0]):
            assert np.all(out[:, q, :] == out[:, q, :1])
            assert np.all(np.abs(out[:, q, 0] - ref[:, row]) <= (0 if v[0, 0, 0] == int(v[0, 0, 0]) else 5 * U * mag[:, row]))
