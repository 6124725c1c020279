"""Bounded waits on mbarriers where a warp goes on together, from the sources:
the lanes of a warp can end a bounded wait differently (one sees that another
role has given up, its neighbour sees the phase complete), and a lane that
leaves a loop alone leaves the others at the loop's warp barrier.  So a wait
outside a role of one lane is put to the warp's vote."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2101_12597_gb300", "csrc")
FILES = sorted(p for ext in ("*.cu", "*.cuh") for p in glob.glob(os.path.join(CSRC, ext)))


def unvoted(source):
    """(line number, line) of every mbar_wait whose enclosing blocks and statement
    neither select one lane nor vote."""
    source = re.sub(r"//[^\n]*", "", source)
    stack, stmt, found, line = [], "", [], 1
    for i, ch in enumerate(source):
        if ch == "{":
            stack.append(stmt)
            stmt = ""
        elif ch == "}":
            stack.pop()
            stmt = ""
        elif ch == ";" and stmt.count("(") == stmt.count(")"):
            stmt = ""
        else:
            stmt += ch
        if source.startswith("mbar_wait(", i) and not re.match(r"\w", source[i - 1]):
            where = stack + [stmt]
            if not any("lane == 0" in s or "__all_sync(" in s for s in where) \
                    and "bool" not in stmt.split()[-2:]:
                found.append((line, source[i:].split("\n")[0]))
        line += ch == "\n"
    return found


def test_the_scan_sees_an_unvoted_wait():
    assert unvoted("void f() { if (w) { for (;;) { if (use && !mbar_wait(&b, 0)) break; } } }")
    assert not unvoted("void f() { if (lane == 0) { mbar_wait(&b, 0); } }")
    assert not unvoted("void f() { ok = __all_sync(~0u, mbar_wait(&b, 0)); }")
    assert not unvoted("void f() { if (!mbar_wait_warp(&b, 0)) return; }")


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_waits_of_whole_warps_are_voted(path):
    bad = unvoted(open(path).read())
    assert not bad, bad
