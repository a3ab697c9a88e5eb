"""Bounded waits of the kernels whose warps have roles, read from their sources: a wait that gives up
must not split a warp in front of a warp-collective instruction (TMEM access, barrier) or leave other
warps in a barrier that no longer fills. So a wait by a whole warp goes through warp_wait, a plain
mbar_wait stands in a branch of one thread or only sets a flag of its thread, and warps that meet in a barrier of their role do not leave
their loop in between: either the barrier carries the outcome of their waits, or no wait jumps out."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_10377_gb300", "csrc")
ROLES = ["k_project_tc.cu", "k_project_tc32.cu", "k_project_bwd_tc.cu", "k_project_bwd_tc32.cu", "k_gradfeat.cu"]
ONE_THREAD = re.compile(r"\b(lane|tid|threadIdx\.x) == 0\b|\bissue_by_one_thread\(")


def _enclosing_blocks(src):
    """For every plain wait: its line number and the headers of the braces around it."""
    src = re.sub(r"//[^\n]*", "", src)
    src = re.sub(r"\bif \(ok\) ok = tc::mbar_wait", "keep_going", src)     # no branch depends on the outcome
    stack, start, found = [], 0, []
    for m in re.finditer(r"[{};]|\bmbar_wait(_cluster)?\(", src):
        t = m.group()
        if t == "{":
            stack.append(src[start:m.start()])
        elif t == "}":
            stack.pop()
        elif t != ";":
            found.append((src.count("\n", 0, m.start()) + 1, list(stack)))
            continue
        start = m.end()
    return found


@pytest.mark.parametrize("name", ROLES)
def test_plain_waits_stand_in_branches_of_one_thread(name):
    waits = _enclosing_blocks(open(os.path.join(CSRC, name)).read())
    assert [line for line, blocks in waits if not any(ONE_THREAD.search(h) for h in blocks)] == []


@pytest.mark.parametrize("name", ROLES)
def test_no_wait_jumps_past_a_role_barrier(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for role in re.split(r"\n  } else(?: if \([^\n]*)? \{", src):      # the branches of the kernel's role dispatch
        if "named_barrier_sync" in role:
            assert not re.search(r"if \(!tc::\w*wait\w*\([^\n]*(goto|break|return)", role)
