"""Properties of the tcgen05 kernel's source that no run shows: what only
matters after a wait has run out, and orderings between the two CTAs of a pair
that hold on one machine by chance."""
import os
import re
import subprocess

from paper_2608_21229_gb300 import build as cbuild

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


def test_waits_for_the_other_ctas_stores_and_reads_are_at_cluster_scope():
    """The follower's E4M3 Q tile is written, and the item ring read, with
    ordinary instructions: the arrivals release, and the leader's waits acquire,
    at cluster scope (an mbarrier operation without a scope is at CTA scope)."""
    code, ptx = _code("attn_tc2.cuh"), _code("ptx.cuh")
    for name, op in (("mbar_arrive_release_cluster", "mbarrier.arrive.release.cluster"),
                     ("mbar_try_wait_acquire_cluster", "try_wait.parity.acquire.cluster")):
        assert op in ptx[ptx.index(name):][:400]
    for line in code.splitlines():
        if "mbar_arrive" in line and ("kQ8Full" in line or "kItemEmpty" in line):
            assert "mbar_arrive_release_cluster" in line, line
        if "wait_" in line and ("kQ8Full" in line or "kItemEmpty" in line):
            assert "wait_cl_acquire" in line, line
    assert sum("wait_cl_acquire" in line for line in code.splitlines()) >= 4
    helper = code[code.index("bool wait_cl_acquire("):][:300]
    assert "mbar_try_wait_acquire_cluster" in helper


def test_the_kernel_behind_may_start_only_after_the_wait_for_the_one_before():
    """The cache writes, dependents of the prefill, start on its triggers and wait
    for nothing themselves before they write the cache: so a CTA triggers only
    after its own wait, on every path."""
    code = _code("attn_tc2.cuh")
    kernel = code[code.index("attn_tc2_kernel("):]
    assert kernel.count("grid_dependency_wait()") == 1 and kernel.count("grid_launch_dependents()") == 1
    assert kernel.index("grid_dependency_wait()") < kernel.index("grid_launch_dependents()")


def test_pair_kernel_keeps_no_arrays_in_local_memory(tmp_path):
    """The roles' state lives in registers: an array indexed at run time goes to
    local memory, where the producer of the E4M3 kernel spent more time than a
    small step takes.  (A spilled register or two is no such array.)"""
    cmd = cbuild.nvcc_cmd(str(tmp_path / "x.so"), ["-Xptxas", "-v"])
    log = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
    frames = dict(re.findall(r"Function properties for (\S*attn_tc2_kernel\S*)\s+(\d+) bytes stack frame", log))
    assert len(frames) == 5, sorted(frames)
    assert all(int(n) <= 16 for n in frames.values()), frames
