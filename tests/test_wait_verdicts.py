"""A wait that may give up has one verdict per warp wherever the warp goes on together (tcgen05, ldmatrix, stmatrix, mma
and elect take all 32 lanes): the helpers that answer each lane for itself are called in code of a single thread or
inside a vote.  Read from the sources: on a GPU only a wait that runs out would show a violation."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_00288_b200", "csrc")
PER_LANE = re.compile(r"\b(mbar_wait_bounded|mbar_wait_a|mbar_spin_a|mbar_test_a)\s*\(")
ONE_THREAD = re.compile(r"\b(lane|tid|threadIdx\.x) == 0\b")


def _without_comments(text):
    return re.sub(r"//[^\n]*", "", text)


def _enclosing_heads(text, at):
    """What stands before each brace that is open at `at`, innermost first."""
    heads, depth = [], 0
    for i in range(at - 1, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth:
                depth -= 1
                continue
            start = max(text.rfind(c, 0, i) for c in ";{}")
            heads.append(text[start + 1:i])
    return heads


@pytest.mark.parametrize("name", ["forward.cu", "wgrad.cu"])
def test_waits_of_whole_warps_are_voted(name):
    text = _without_comments(open(os.path.join(CSRC, name)).read())
    uses = list(PER_LANE.finditer(text))
    assert len(uses) + len(re.findall(r"\b(?:mbar_wait_warp|mbar_wait_warp_a)\s*\(", text)) >= 5
    for use in uses:
        statement = text[max(text.rfind(c, 0, use.start()) for c in ";{}") + 1:use.start()]
        single = any(ONE_THREAD.search(h) for h in _enclosing_heads(text, use.start()))
        # (an epilogue without store warps goes by its leader's answer, which it publishes at the group's barrier: it picks the
        # helper by its form)
        by_form = re.search(r"const bool got = (kStoreWarps|RES) \? mbar_wait_warp\(", statement)
        assert single or by_form or "__all_sync(" in statement, f"{name}: {text[use.start() - 60:use.end() + 60]}"
