"""Hand-overs through shared memory, checked in the kernels' source.

A write after a read that lacks its barrier shows in no run (a converged warp
reads with one instruction), so it is looked for where it is written.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0810_4737_gb300", "csrc")


def _function(name, text):
    """The body of a function: from its name to the brace that closes it."""
    start = text.index("{", text.index(")\n", text.index(name)))
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return re.sub(r"//[^\n]*", "", text[start:i + 1])
    raise AssertionError(name)


def test_a_track_s_source_is_not_read_where_the_next_one_s_is_written():
    """In the one-warp kernel lane 0 writes S->src as soon as it asks for the
    next track: every read by the other lanes has its barrier before that."""
    with open(os.path.join(CSRC, "reed_ion.cuh")) as f:
        text = f.read()
    assert "S->src" not in _function("int follow_track(", text)
    # acquire_track: behind the barrier that follows lane 0's block, and the caller
    # starts a track (with barriers of its own) or ends
    body = _function("int acquire_track(", text)
    lane0, rest = body.split("    __syncwarp();\n    const int src = S->src;\n", 1)
    assert lane0.index("if (lane == 0) {") < lane0.index("S->src") and "S->src" not in rest
    # the loop over tracks: read between two barriers, in both forms of the kernel
    body = _function("reed_ion_kernel(", text)
    assert len(re.findall(r"S->src\b", body)) == 1
    assert re.search(r"if \(ADJ\) __syncthreads\(\);\s*const int src = S->src;\s*if \(!ADJ\) __syncwarp\(\);", body)
    assert re.search(r"__syncthreads\(\);\s*}\s*}\s*if \(tid == 0\)", body)   # (ADJ: at the loop's end)
