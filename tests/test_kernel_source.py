"""Properties of the tcgen05 kernel's source that no run shows: what only
matters after a wait has run out, and orderings between the two CTAs of a pair
that hold on one machine by chance."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_21229_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _guard_of(code, at):
    """The condition of the innermost if-block around position `at` that tests a lane."""
    depth, i = 0, at
    while i > 0:
        i -= 1
        if code[i] == "}":
            depth += 1
        elif code[i] == "{":
            if depth:
                depth -= 1
                continue
            head = code[code.rfind("\n", 0, i) + 1:i]
            if "elect_one()" in head or "lane ==" in head:
                return head.strip()
    return None


def test_every_commit_is_issued_by_the_lane_that_issued_the_mmas():
    """tcgen05.commit tracks the executing thread's own MMAs.  The MMAs run
    under elect.sync, whose lane PTX leaves open, so the commit that the freeing
    of tensor memory waits for has to be issued under elect.sync as well."""
    code = _code("attn_tc2.cuh")
    at = [m.start() for m in re.finditer(r"tc2_commit_mc\(", code)]
    assert len(at) >= 5
    guards = [_guard_of(code, i) for i in at]
    direct = [g for g in guards if g is not None]  # (commits inside the issue_* lambdas have none of their own)
    assert direct and all("elect_one()" in g and "lane ==" not in g for g in direct), direct
    done = code[code.index("mma_done:"):code.index("drain_one(bar(L::kMmaDone)")]
    assert "elect_one()" in done and "__syncwarp()" in done
