"""The climb of the upward pass, read as text: one lane arrives at a parent with an acquire-release atomic, then
every lane of its warp may read what the sibling's warp wrote.  Ballots and shuffles order no memory
between lanes, so a warp barrier has to stand between the arrival and the lanes' reads on every
iteration, and one between the lanes' stores and the arrival that publishes them.  No run can show
its absence reliably, so this looks at the kernel's loop itself."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _climb():
    """The body of k_upward's climbing loop, without comments."""
    with open(os.path.join(ROOT, "paper_1609_08621_gb300", "csrc", "tree.cu")) as f:
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
    at = src.index("for (;;) {", src.index("k_upward(")) + len("for (;;) {")
    depth, end = 1, at
    while depth:
        depth += {"{": 1, "}": -1}.get(src[end], 0)
        end += 1
    return src[at:end - 1]


def _unconditional(text):
    """text without its nested blocks and without statements that an `if` on the same line guards."""
    out, depth = [], 0
    for ch in text:
        depth += {"{": 1, "}": -1}.get(ch, 0)
        if depth == 0:
            out.append(";" if ch == "}" else ch)
    return re.sub(r"\bif\s*\([^;]*;", "", "".join(out))


def test_barriers_around_the_arrival():
    body = _climb()
    arrival = body.index("arrive_acq_rel(")
    statement_end = body.index(";", arrival) + 1
    readers = [body.index(f) for f in ("up_cell_thread(", "up_cell_warp(")]
    assert all(r > statement_end for r in readers)
    assert "__syncwarp();" in _unconditional(body[:body.rindex(";", 0, arrival) + 1])
    between = body[statement_end:min(readers)]
    assert "__syncwarp();" in _unconditional(between), between
