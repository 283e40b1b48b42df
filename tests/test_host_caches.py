"""Values that the launch functions keep per device (attributes set, grids found) are shared by
every calling thread: each such function-local static is a std::atomic, and a cache of a value
and a flag is one atomic word, so that no thread sees the flag without the value."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_01990_gb300", "csrc")


def test_function_local_caches_are_atomic():
    plain, atomic = [], {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"^[ \t]+static (?!constexpr|const |_?assert)([\w:<>]+) (\w+)(\[\d+\])?\s*(=[^;]*)?;", text, re.M):
            if m.group(1).startswith("std::atomic"):
                atomic.setdefault(os.path.basename(path), []).append(m.group(2))
            else:
                plain.append((os.path.basename(path), m.group(2)))
    assert not plain, plain
    assert sorted(atomic["tdc_sytrd.cu"]) == ["attr", "grid", "known"] and atomic["tdc_banded.cu"] == ["attr"]
