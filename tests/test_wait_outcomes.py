"""A bounded wait may run out in some lanes of a warp and not in others, and what a whole warp does together (votes, shuffles, warp
barriers, tensor-memory loads) has no limit of its own: a lane that left its loop alone would hold the others there for good.
So a kernel waits in one lane only, or as a warp (mbar_wait_warp), or a vote on the outcome comes before any lane leaves on it.  Read
from the sources: no GPU run can bring such a mixed outcome about without the risk that it stands for."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_18753_b200", "csrc")
WAIT = re.compile(r"\b(wait_on|mbar_wait|mbar_wait_cluster)\(")
HELPER = re.compile(r"auto wait_(on|all) = ")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", lambda m: " " * len(m.group()), text)


def _in_one_lane(text, at):
    """Whether a brace around position `at` was opened by a condition on lane 0."""
    depth = 0
    for k in range(at, -1, -1):
        if text[k] == "}":
            depth += 1
        elif text[k] == "{":
            if depth:
                depth -= 1
            elif re.search(r"if \(lane == 0[^{]*$", text[text.rfind("\n", 0, k) + 1:k]):
                return True
    return False


def _unvoted(text):
    bad = []
    for m in WAIT.finditer(text):
        line = text[text.rfind("\n", 0, m.start()) + 1:text.find("\n", m.start())]
        if HELPER.search(line) or _in_one_lane(text, m.start()):
            continue
        # kept in a variable: on its way to the vote no lane may leave
        got = re.match(r"\s*(?:if \([^;]*\) )?(?:const bool |bool )?(\w+) = ", line)
        rest = text[m.end():]
        vote = re.search(r"__a(ll|ny)_sync\([^;]*\b%s\b" % got.group(1), rest) if got else None
        if vote is None or re.search(r"\b(break|return|continue)\b", rest[:vote.start()]):
            bad.append(line.strip())
    return bad


@pytest.mark.parametrize("name", [f for f in sorted(os.listdir(CSRC)) if WAIT.search(_source(f)) and f != "sm100_ptx.cuh"])
def test_no_lane_acts_on_its_own_outcome(name):
    assert _unvoted(_source(name)) == []


def test_the_reader_finds_a_lane_that_leaves_alone():
    """What the check is for, planted: a wait of every lane, left by those whose limit ran out."""
    assert _unvoted("{\n  ok = wait_on(bar(FULL), 0);\n  if (!ok) break;\n  any = __any_sync(0xffffffffu, any);\n}")
    assert not _unvoted("{\n  const bool here = wait_on(bar(FULL), 0);\n  ok = __all_sync(0xffffffffu, here);\n  if (!ok) break;\n}")
    assert not _unvoted("{\n  ok = ptx::mbar_wait_warp(bar(FULL), 0, abort_flag);\n  if (!ok) break;\n}")
    assert not _unvoted("if (lane == 0) {\n  ok = wait_on(bar(FULL), 0);\n  if (!ok) break;\n}")
