"""Performance cases: what users of this library have it do, through its public calls.

Every case is one call of an entry point of ``paper_2008_01990_gb300.tdc`` (for the adjoint, a
forward and a backward pass through autograd).  The sizes are those of the repository's tests
and benchmark, or lie between them, odd ones among them.  ``listed`` names the standing cases,
``draw`` gives further ones of the same ranges.

Matrix families (the spectra differ in how much a merge deflates and in the ranks of the
eigenvector matrices' off-diagonal tiles):

* ``uniform``  d, e uniform(-1, 1): localised eigenvectors, nearly everything deflates;
* ``chain``    d = 2 + a ramp + weak disorder, e = 1: a one-dimensional discretised operator in
               a smooth potential, extended eigenvectors, almost nothing deflates;
* ``hermite``  d constant, e_i = sqrt(i + mu): the recurrence of the (associated) Hermite
               polynomials, whose eigenproblem gives Gauss quadrature nodes and weights.
"""
import math

import numpy as np
import torch

from paper_2008_01990_gb300 import tdc

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # A small problem, as one calls it in a loop: launches and latency decide.
        {"name": "eig_small", "kind": "eig", "family": "uniform", "n": 300},
        # The order of the accuracy tests and of the benchmark's first configuration.
        {"name": "eig_1024", "kind": "eig", "family": "uniform", "n": 1024},
        # Nodes and weights of a Gauss rule (odd order, smooth eigenvectors, no deflation).
        {"name": "eig_gauss_4999", "kind": "eig", "family": "hermite", "n": 4999},
        # The headline order: all eigenvectors of a discretised one-dimensional operator.
        {"name": "eig_16384", "kind": "eig", "family": "chain", "n": 16384},
        # Many independent problems of mixed orders in one call.
        {"name": "batched_512", "kind": "batched", "count": 512, "lo": 64, "hi": 1024},
        # A training step through the eigen-decomposition: forward and adjoint of a batch.
        {"name": "adjoint_256x512", "kind": "adjoint", "count": 256, "n": 512},
        # Dense symmetric matrices: reduction, divide and conquer, back-transform.
        {"name": "syevd_1000", "kind": "syevd", "n": 1000},
        {"name": "syevd_4096", "kind": "syevd", "n": 4096},
        # A symmetric band matrix (finite differences of high order, coupled chains).
        {"name": "sbevd_2048_b8", "kind": "sbevd", "n": 2048, "b": 8},
        # The SVD of a bidiagonal matrix (second half of a dense SVD), odd order.
        {"name": "bdsdc_3001", "kind": "bdsdc", "n": 3001},
        # The structured matrix product on its own (Example 1 of the paper, its first order).
        {"name": "cauchy_8192", "kind": "cauchy", "m": 8192, "n": 8192, "mode": "structured_split"},
        # A product with a Toeplitz operand (filtering many signals), split precision.
        {"name": "toeplitz_4096", "kind": "operand", "operand": "toeplitz", "m": 4096, "n": 4096, "mode": "split"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eig", "eig", "eig", "batched", "adjoint", "syevd", "syevd", "sbevd", "bdsdc", "cauchy",
                       "operand"])
    if kind == "eig":
        family = rng.choice(["uniform", "chain", "hermite"])
        n = _log_int(rng, 50, 1500 if family == "uniform" else 12000)
        return {"kind": kind, "family": family, "n": n}
    if kind == "batched":
        lo = rng.choice([17, 64, 100])
        return {"kind": kind, "count": _log_int(rng, 16, 400), "lo": lo, "hi": _log_int(rng, 2 * lo, 1024)}
    if kind == "adjoint":
        return {"kind": kind, "count": _log_int(rng, 4, 256), "n": _log_int(rng, 60, 512)}
    if kind == "syevd":
        return {"kind": kind, "n": _log_int(rng, 200, 4000)}
    if kind == "sbevd":
        return {"kind": kind, "n": _log_int(rng, 300, 2500), "b": rng.choice([2, 3, 5, 8, 16])}
    if kind == "bdsdc":
        return {"kind": kind, "n": _log_int(rng, 150, 4000)}
    if kind == "cauchy":
        mode = rng.choice(["dense", "split", "structured_split", "structured_split"])
        lo, hi = {"dense": (100, 1500), "split": (200, 5000), "structured_split": (1500, 8192)}[mode]
        return {"kind": kind, "m": _log_int(rng, lo, hi), "n": _log_int(rng, lo, hi), "mode": mode}
    operand = rng.choice(["toeplitz", "hankel", "dft"])
    mode = rng.choice(["dense", "split", "split"])
    hi = 1000 if mode == "dense" else 4000
    return {"kind": kind, "operand": operand, "m": _log_int(rng, 150, hi), "n": _log_int(rng, 150, hi), "mode": mode}


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, dtype=F64, device=DEV, generator=g) * (hi - lo) + lo


def _colmajor(g, m, n, lo, hi):
    return _uniform(g, n, m, lo=lo, hi=hi).t()


def _tridiagonal(family, n, g):
    if family == "uniform":
        return _uniform(g, n, lo=-1.0, hi=1.0), _uniform(g, n - 1, lo=-1.0, hi=1.0)
    c = float(_uniform(g, 1, lo=0.4, hi=0.6))
    if family == "chain":
        x = torch.arange(n, dtype=F64, device=DEV) / n
        return 2.0 + c * x + 1e-3 * _uniform(g, n, lo=-1.0, hi=1.0), torch.ones(n - 1, dtype=F64, device=DEV)
    i = torch.arange(1, n, dtype=F64, device=DEV)
    return torch.full((n,), c, dtype=F64, device=DEV), torch.sqrt(i + c)


def _weak_disorder(count, n, g):
    """Rows of extended problems with well separated eigenvalues, as an adjoint needs them."""
    x = torch.arange(n, dtype=F64, device=DEV) / n
    d = _uniform(g, count, 1, lo=0.3, hi=1.0) * x + _uniform(g, count, n, lo=-0.05, hi=0.05)
    return d, 1.0 + _uniform(g, count, n - 1, lo=-0.05, hi=0.05)


def _sizes(case):
    r = np.random.RandomState(case["count"])
    return r.randint(case["lo"], case["hi"] + 1, case["count"]).astype(np.int64)


def _dense_symmetric(n, g):
    x = _uniform(g, n, n, lo=-1.0, hi=1.0)
    return 0.5 * (x + x.t())


def _band(n, b, g):
    ab = _uniform(g, b + 1, n, lo=-1.0, hi=1.0)
    for r in range(1, b + 1):
        ab[r, n - r:] = 0.0
    return ab


def _bidiagonal(n, g):
    sign = torch.where(_uniform(g, n) < 0.5, -1.0, 1.0).to(F64)
    return _uniform(g, n, lo=0.5, hi=1.5) * sign, _uniform(g, n - 1, lo=-1.0, hi=1.0)


def _example1(n, g):
    i = torch.arange(1, n + 1, dtype=F64, device=DEV)
    d = i * (8.0 / n)
    return d, d + 4.0 / n, _uniform(g, n), _uniform(g, n)


_MODES = {"dense": tdc.MERGE_DENSE, "split": tdc.MERGE_SPLIT, "structured_split": tdc.MERGE_STRUCTURED_SPLIT}
_OPERANDS = {"toeplitz": tdc.TOEPLITZ, "hankel": tdc.HANKEL}


def _inputs(case, seed):
    """The call's inputs alone, the same for the library and for the exact values."""
    g, kind = _gen(seed), case["kind"]
    if kind == "eig":
        return _tridiagonal(case["family"], case["n"], g)
    if kind == "batched":
        total = int(_sizes(case).sum())
        return _uniform(g, total, lo=-1.0, hi=1.0), _uniform(g, total, lo=-1.0, hi=1.0)
    if kind == "adjoint":
        count, n = case["count"], case["n"]
        d, e = _weak_disorder(count, n, g)
        w = torch.randn(count, n, dtype=F64, device=DEV, generator=g)
        return d, e, w, torch.randn(count, n, n, dtype=F64, device=DEV, generator=g)
    if kind == "syevd":
        return (_dense_symmetric(case["n"], g),)
    if kind == "sbevd":
        return (_band(case["n"], case["b"], g),)
    if kind == "bdsdc":
        return _bidiagonal(case["n"], g)
    if kind == "cauchy":
        return (_colmajor(g, case["m"], case["n"], -1.0, 1.0),) + _example1(case["n"], g)
    a = _colmajor(g, case["m"], case["n"], -1.0, 1.0)
    return (a,) if case["operand"] == "dft" else (a, _uniform(g, 2 * case["n"] - 1, lo=-1.0, hi=1.0))


def prepare(case, seed):
    s = {"case": case, "in": _inputs(case, seed)}
    kind = case["kind"]
    if kind == "eig":
        n = case["n"]
        s["ws"] = tdc.workspace(tdc.workspace_size(n))
        s["lam"] = torch.empty(n, dtype=F64, device=DEV)
        s["Q"] = torch.empty(n, n, dtype=F64, device=DEV).t()
    elif kind == "batched":
        sizes = _sizes(case)
        s["sizes"] = sizes
        s["off_de"] = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.int64)
        s["off_q"] = np.concatenate([[0], np.cumsum(sizes * sizes)[:-1]]).astype(np.int64)
        s["ws"] = tdc.workspace(tdc.batched_workspace_size(sizes))
        s["lam"] = torch.empty(int(sizes.sum()), dtype=F64, device=DEV)
        s["Q"] = torch.empty(int((sizes * sizes).sum()), dtype=F64, device=DEV)
    elif kind == "adjoint":
        d, e, w, gq = s["in"]
        s["in"] = (d.requires_grad_(), e.requires_grad_(), w, gq)
    elif kind == "syevd":
        s["ws"] = tdc.workspace(tdc.syevd_workspace_size(case["n"]))
    return s


def run(s):
    case, x = s["case"], s["in"]
    kind = case["kind"]
    if kind == "eig":
        return tdc.eig(x[0], x[1], ws=s["ws"], lam=s["lam"], Q=s["Q"])
    if kind == "batched":
        return tdc.eig_batched(s["sizes"], x[0], x[1], s["off_de"], s["off_q"], s["lam"], s["Q"], ws=s["ws"])
    if kind == "adjoint":
        d, e, w, gq = x
        lam, q = tdc.eigh_tridiagonal(d, e)
        d_bar, e_bar = torch.autograd.grad((lam, q), (d, e), (w, gq))
        return lam.detach(), d_bar, e_bar, q.detach()
    if kind == "syevd":
        return tdc.syevd(x[0], ws=s["ws"])
    if kind == "sbevd":
        return tdc.sbevd(x[0])
    if kind == "bdsdc":
        return tdc.bdsdc(x[0], x[1])
    if kind == "cauchy":
        return tdc.cauchy_like_gemm(*x, mode=_MODES[case["mode"]])
    if case["operand"] == "dft":
        return tdc.dft_gemm(x[0], mode=_MODES[case["mode"]])
    return tdc.structured_gemm(x[0], x[1], kind=_OPERANDS[case["operand"]], mode=_MODES[case["mode"]])


def work(case):
    """Inputs read once, outputs written once, and the operations of the methods themselves:
    for tridiagonal and band problems with all eigenvectors a few operations per entry of Q,
    for dense ones the reduction (4/3 n^3) and the back-transform (2 n^3), for a product 2 m n
    per column of the operand (the structured product: 4 m n log2 n)."""
    kind = case["kind"]
    if kind == "eig":
        n = case["n"]
        return {"bytes": 8.0 * (n * n + 3 * n), "flops": 10.0 * n * n}
    if kind == "batched":
        mean_sq = (case["hi"] ** 3 - case["lo"] ** 3) / (3.0 * max(case["hi"] - case["lo"], 1))
        return {"bytes": 8.0 * case["count"] * mean_sq, "flops": 10.0 * case["count"] * mean_sq}
    if kind == "adjoint":
        c, n = case["count"], case["n"]
        return {"bytes": 8.0 * c * (2 * n * n + 6 * n), "flops": c * 4.0 * n ** 3}
    if kind == "syevd":
        n = case["n"]
        return {"bytes": 16.0 * n * n, "flops": 10.0 / 3.0 * n ** 3}
    if kind == "sbevd":
        n, b = case["n"], case["b"]
        return {"bytes": 8.0 * (n * n + (b + 2) * n), "flops": 10.0 * b * n * n}
    if kind == "bdsdc":
        n = case["n"]
        return {"bytes": 8.0 * (2 * n * n + 3 * n), "flops": 20.0 * n * n}
    m, n = case["m"], case["n"]
    if kind == "cauchy":
        flops = 4.0 * m * n * math.log2(n) if case["mode"] == "structured_split" else 2.0 * m * n * n
        return {"bytes": 8.0 * (2 * m * n + 4 * n), "flops": flops}
    two = 2 if case["operand"] == "dft" else 1
    return {"bytes": 8.0 * ((1 + two) * m * n + 2 * n), "flops": 2.0 * two * m * n * n}


def _positive(*parts):
    """Columns scaled by +-1 so that the entry of largest magnitude over all parts is positive."""
    whole = torch.cat(parts, dim=-2)
    top = whole.gather(-2, whole.abs().argmax(dim=-2, keepdim=True))
    sign = torch.where(top < 0, -1.0, 1.0).to(F64)
    return tuple(p * sign for p in parts)


def _eigh_tridiagonal(d, e):
    lam, q = torch.linalg.eigh(torch.diag_embed(d) + torch.diag_embed(e, 1) + torch.diag_embed(e, -1))
    return lam, _positive(q)[0]


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "eig":
        return _eigh_tridiagonal(*x) if case["n"] <= 8192 else None
    if kind == "batched":
        d, e, at, lam, q = x[0], x[1], 0, [], []
        for n in _sizes(case):
            n = int(n)
            if len(lam) >= 700:
                return None
            v, u = _eigh_tridiagonal(d[at:at + n], e[at:at + n - 1])
            lam.append(v)
            q.append(u.t().reshape(-1))
            at += n
        return torch.cat(lam), torch.cat(q)
    if kind == "adjoint":
        d, e, w, gq = x
        out = []
        for k in range(case["count"]):
            lam, q = _eigh_tridiagonal(d[k], e[k])
            gap = lam[None, :] - lam[:, None]
            f = torch.where(gap == 0, 0.0, 1.0 / torch.where(gap == 0, 1.0, gap))
            p = q.t() @ gq[k]
            t = q @ (torch.diag(w[k]) + f * (0.5 * (p - p.t()))) @ q.t()
            out.append((lam, torch.diagonal(t), 2.0 * torch.diagonal(t, 1), q))
        return tuple(torch.stack(v) for v in zip(*out))
    if kind == "syevd":  # the columns' signs go by the reduction: the vectors have no value of their own
        return torch.linalg.eigvalsh(x[0]), None
    if kind == "sbevd":
        ab = x[0]
        full = torch.diag(ab[0])
        for r in range(1, case["b"] + 1):
            low = torch.diag(ab[r, :case["n"] - r], -r)
            full = full + low + low.t()
        return torch.linalg.eigvalsh(full), None
    if kind == "bdsdc":
        u, sigma, vt = torch.linalg.svd(torch.diag(x[0]) + torch.diag(x[1], 1))
        v, u = _positive(vt.t(), u)
        return sigma, u, v.t()
    if kind == "cauchy":
        a, d, w, u, v = x
        return a @ (u[:, None] * v[None, :] / (d[:, None] - w[None, :]))
    a, n = x[0], case["n"]
    k = torch.arange(n, device=DEV)
    if case["operand"] == "dft":
        angle = ((k[:, None] * k[None, :]) % n).to(F64) * (2.0 * math.pi / n)
        return a @ torch.cos(angle), -(a @ torch.sin(angle))
    at = k[:, None] - k[None, :] + n - 1 if case["operand"] == "toeplitz" else k[:, None] + k[None, :]
    return a @ x[1][at]
