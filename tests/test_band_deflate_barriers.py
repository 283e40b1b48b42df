"""The band deflation's lists cross threads: each is written by the thread of one index and
read by the threads of others, so a block barrier at the kernel's own level (not inside the
loop that wrote it) has to lie between the writing loop and the first reading one.  Walked
through in the kernel's source, as a missing barrier cannot be shown safely by running it."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_01990_gb300", "csrc",
                   "tdc_banded.cu")


def kernel_body(text, name):
    text = re.sub(r"//[^\n]*", "", text)
    at = text.index("{", text.index(name + "(BdLevel L)"))
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at + 1:i]
        i += 1


def events(body, array):
    """('w' | 'r' | 'b', position): writes and reads of array[...], and barriers at depth 0."""
    out = []
    for m in re.finditer(r"\b%s\[[^\]]*\](\s*=(?!=))?" % array, body):
        out.append((m.start(), "w" if m.group(1) else "r"))
    for m in re.finditer(r"__syncthreads\(\);", body):
        before = body[:m.start()]
        if before.count("{") == before.count("}"):
            out.append((m.start(), "b"))
    return [k for _, k in sorted(out)]


def crossing(ev):
    """Whether some read follows a write without a barrier in between."""
    open_write = False
    for k in ev:
        open_write = True if k == "w" else (False if k == "b" else open_write)
        if k == "r" and open_write:
            return True
    return False


@pytest.mark.parametrize("array", ["surv", "rotbit", "rc", "rs", "rw", "rdp", "rdn"])
def test_lists_are_complete_before_they_are_read(array):
    ev = events(kernel_body(open(SRC).read(), "k_bd_deflate"), array)
    assert "w" in ev and "r" in ev and not crossing(ev), ev


def test_a_missing_barrier_is_found():
    body = kernel_body(open(SRC).read(), "k_bd_deflate")
    at = body.index("__syncthreads();", body.index("surv[M + pos] ="))
    assert crossing(events(body[:at] + body[at + len("__syncthreads();"):], "surv"))
