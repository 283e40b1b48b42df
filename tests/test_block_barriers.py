"""Barriers that a block's warps depend on, walked through in the kernels' sources (a missing one
cannot be shown safely by running it)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_01990_gb300", "csrc")


def body_after(text, start):
    """The braced body that follows `start`, without comments."""
    text = re.sub(r"//[^\n]*", "", text)
    at = text.index("{", text.index(start))
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at + 1:i]
        i += 1


def source(name):
    return open(os.path.join(CSRC, name)).read()


def shared_exit_flags(body):
    """Loop conditions that read shared memory which the loop itself writes: one warp may already
    have set it in the next round when another evaluates the condition."""
    found = []
    for m in re.finditer(r"\bwhile \(!?(\w+)\[(\w+)\]\)\s*\{", body):
        inner = body_after(body[m.start():], "while")
        if re.search(r"\b%s\[%s\]\s*=(?!=)" % (m.group(1), m.group(2)), inner):
            found.append(m.group(0))
    return found


def test_leaf_iteration_ends_at_a_barrier():
    """The two warps of a leaf leave the QR iteration together: its end comes out of the barrier."""
    body = body_after(source("tdc_merge.cu"), "k_leaf(Plan P, int64_t nleaves)")
    assert shared_exit_flags(body) == []
    assert re.search(r"last = __syncthreads_or\(end \? 1 : 0\) != 0;\s*\+\+sweep;\s*\}", body)


def test_a_shared_exit_flag_is_found():
    body = "ctrl[4] = 0; __syncthreads(); while (!ctrl[4]) { if (warp == 0) ctrl[4] = 1; __syncthreads(); }"
    assert len(shared_exit_flags(body)) == 1


def test_fp64_tiles_meet_before_their_columns_are_stored():
    """A tile's column places and scales, written by its first threads, are read by all in the epilogue:
    the pole loop's barriers lie in between, and where the half has no pole a barrier of its own."""
    body = body_after(source("tdc_gemm_dense.cu"), "void dense_tile(")
    write, read = body.index("sc.Pos[tid] ="), body.index("const int pos = sc.Pos[")
    between = body[write:read]
    assert "for (int k0 = qlo; k0 < qhi; k0 += BK) {" in between
    after_loop = between[between.index("for (int k0 = qlo"):]
    assert re.search(r"if \(qlo >= qhi\) __syncthreads\(\);", after_loop)


def test_split_segments_are_kept_and_counted_alike():
    """The split path's list holds exactly the merge parts whose output tiles its offsets count: a part
    without a pole (no digit images) has output tiles too, and skipping it would leave its rows unwritten
    and tiles that belong to no segment."""
    body = body_after(source("tdc_gemm_split.cu"), "k_split_segs(Plan P, int level")
    assert re.search(r"cns \+= tt > 0 \? 1 : 0;", body) and re.search(r"if \(tt == 0\) continue;", body)
    assert not re.search(r"if \(el == 0\) continue", body)
