"""Rules of the tensor-core kernels that no run can show, read from their source: a bounded wait may run out in one warp and complete
in the next, so warps that meet in a barrier afterwards must leave together or not at all.  A kernel that got this wrong would hang,
and only after another fault had raised its abort flag."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_20407_b200", "csrc")
TOKENS = re.compile(r"\b(mbar_wait|named_barrier_all|named_barrier|cluster_sync|break|continue|return)\b")


def tokens(name):
    """(line, token) of everything that waits, meets or leaves, comments and definitions left out; one list per warp role."""
    roles = [[]]
    for number, line in enumerate(open(os.path.join(CSRC, name)), 1):
        if "// -----" in line:                     # a heading: the roles of a kernel, or the parts of a file
            roles.append([])
        for t in TOKENS.findall(re.sub(r"//.*", "", line)):
            roles[-1].append((number, t))
    return [r for r in roles if r]


@pytest.mark.parametrize("name", ["fwd_tc.cu", "bwd_tc.cu"])
def test_warps_that_meet_in_a_barrier_after_a_bounded_wait_decide_together_whether_to_leave(name):
    met = 0
    for role in tokens(name):
        meets = [n for n, (_, t) in enumerate(role) if t == "named_barrier"]
        if not meets:
            continue
        met += 1
        last_wait = max((n for n in range(meets[0]) if role[n][1] == "mbar_wait"), default=None)
        if last_wait is None:
            continue
        between = [t for _, t in role[last_wait + 1:meets[0]]]
        if "named_barrier_all" in between:         # one decision for all of them, and nobody leaves before it
            between = between[:between.index("named_barrier_all")]
        leaving = [t for t in between if t in ("break", "continue", "return")]
        assert not leaving, f"{name}:{role[last_wait][0]}: a warp whose wait ran out leaves, the others wait for it in the barrier at line {role[meets[0]][0]}"
    assert met == 1, f"{name}: {met} roles with a named barrier (this test knows one)"
