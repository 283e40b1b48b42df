"""Calls on another stream than the current one: what a wrapper allocates or copies on the
current stream is waited for and kept alive on the call's stream, for every wrapper, before the
library is entered; what the caller hands in is not touched, and neither is a call on the
current stream.  On the CPU, with stand-ins for the streams and the library."""
import contextlib
import ctypes

import numpy as np
import pytest
import torch

from paper_2008_01990_gb300 import tdc

F64 = torch.float64


class Stream:
    def __init__(self, handle):
        self.cuda_stream = handle
        self.waits = []

    def wait_stream(self, other):
        self.waits.append(other.cuda_stream)


class Library:
    """Every entry point succeeds; the pointers it was given, and what was kept by then."""

    def __init__(self, real, log):
        self.real, self.log = real, log

    def __getattr__(self, name):
        if name.endswith("_size") or name == "tdc_default_opts":
            return getattr(self.real, name)
        log = self.log

        def call(*args):
            log.calls.append((name, {a.value for a in args if isinstance(a, ctypes.c_void_p)}, set(log.kept)))
            return 0
        return call


class Log:
    def __init__(self):
        self.calls, self.kept, self.lent = [], [], None


@pytest.fixture
def log(monkeypatch):
    from paper_2008_01990_gb300 import build
    build.build()
    log = Log()
    real = tdc.lib()
    log.current, log.side, log.capturing = Stream(1), Stream(2), False
    monkeypatch.setattr(tdc, "lib", lambda: Library(real, log))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: log.current)
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda h, *a, **k: log.side if h == 2 else Stream(h))
    monkeypatch.setattr(torch.cuda, "stream", lambda s: contextlib.nullcontext())
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: log.capturing)

    def record(t, s):
        assert s is log.side
        log.kept.append(t.untyped_storage().data_ptr())
    monkeypatch.setattr(torch.Tensor, "record_stream", record)
    return log


def r(*shape):
    return torch.rand(*shape, dtype=F64)


def col(m, n):
    return r(n, m).t()


N = 12
# the wrapper's call, and how many of its own buffers the call takes (outputs, workspace, copies)
CALLS = {
    "eig": (lambda d, **k: tdc.eig(d[0], d[1], **k), 3),
    "rank_one": (lambda d, **k: tdc.rank_one(d[0], d[2], 1.0, **k), 5),
    "cauchy_gemm": (lambda d, **k: tdc.cauchy_gemm(d[3], d[0], torch.zeros(N, dtype=torch.int32), d[0], d[0], d[0], **k), 2),
    "cauchy_like_gemm": (lambda d, **k: tdc.cauchy_like_gemm(d[3], d[0], d[0], d[0], d[0], **k), 2),
    "cauchy_like_ranks": (lambda d, **k: tdc.cauchy_like_ranks(d[0], d[0], d[0], d[0], **k), 2),
    "sytrd": (lambda d, **k: tdc.sytrd(d[3], **k), 5),
    "ormtr": (lambda d, **k: tdc.ormtr(d[3], d[1], d[4], **k), 1),
    "syevd": (lambda d, **k: tdc.syevd(d[3], **k), 4),
    "syevd_overwrite": (lambda d, **k: tdc.syevd(d[3], overwrite=True, **k), 3),
    "structured_gemm": (lambda d, **k: tdc.structured_gemm(d[3], d[5], **k), 2),
    "dft_gemm": (lambda d, **k: tdc.dft_gemm(d[3], **k), 3),
    "sbevd": (lambda d, **k: tdc.sbevd(d[6], **k), 4),
    "bdsdc": (lambda d, **k: tdc.bdsdc(d[0], d[1], **k), 4),
    "eig_backward": (lambda d, **k: tdc.eig_backward(d[0], d[3], d[0], r(N, N), **k), 4),
    "eig_backward_batched": (lambda d, **k: tdc.eig_backward_batched(r(2, N), r(2, N, N), None, r(N, N, 2).permute(2, 0, 1),
                                                                     **k), 4),
}


def data():
    return [r(N), r(N - 1), r(N), col(N, N), col(N, N), r(2 * N - 1), r(3, N)]


@pytest.mark.parametrize("name", sorted(CALLS))
def test_own_buffers_are_kept_and_waited_for(log, name):
    call, own = CALLS[name]
    given = data()
    call(given, stream=log.side)
    work = [c for c in log.calls if c[0] != "tdc_sync_status"]
    assert len(work) == 1 and log.side.waits == [1]
    _, pointers, kept = work[0]
    assert 2 in pointers  # the stream's handle
    assert len(kept & pointers) >= own, (name, len(kept & pointers))
    caller = {t.untyped_storage().data_ptr() for t in given}
    if name not in ("eig_backward",):  # its column-major Q is the caller's when it needs no copy
        assert not kept & caller


def test_batched_workspace(log):
    d = r(2 * N)
    args = ([N, N], d, d, [0, N], [0, N * N], torch.empty(2 * N, dtype=F64), torch.empty(2 * N * N, dtype=F64))
    tdc.eig_batched(*args, stream=log.side)
    assert len(log.kept) == 1 and log.side.waits == [1]
    ws = torch.empty(tdc.batched_workspace_size(np.array([N, N])), dtype=torch.uint8)
    tdc.eig_batched(*args, ws=ws, stream=log.side)
    assert len(log.kept) == 1 and log.side.waits == [1]


def test_nothing_of_the_wrappers_own(log):
    d, e = r(N), r(N - 1)
    ws = torch.empty(tdc.workspace_size(N), dtype=torch.uint8)
    tdc.eig(d, e, ws=ws, lam=torch.empty(N, dtype=F64), Q=col(N, N), stream=log.side)
    assert log.kept == [] and log.side.waits == []


@pytest.mark.parametrize("stream", [None, "current"])
def test_current_stream(log, stream):
    tdc.eig(r(N), r(N - 1), stream=log.current if stream else None)
    assert log.kept == [] and log.current.waits == [] and 1 in log.calls[0][1]


def test_a_capturing_stream_waits_for_nothing_outside(log):
    log.capturing = True
    tdc.eig(r(N), r(N - 1), stream=log.side)
    assert log.side.waits == [] and len(log.kept) == 3
