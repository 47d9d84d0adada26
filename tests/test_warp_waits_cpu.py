"""A bounded wait that runs out must be answered alike by all lanes of a warp wherever the code behind it is the whole warp's
(tensor-memory loads, stmatrix, __syncwarp): a lane that left by itself would be waited for without a limit.  Read from the
sources, because a run that shows it would hang."""
import os
import re

import pytest

from paper_2609_00993_b200 import build as build_mod

# what a whole warp executes together
WHOLE_WARP = r"__syncwarp|__shfl|__all_sync|__ballot|elect_one|tmem_ld|stmatrix|mbar_wait_warp|wait_count"


def _loops(name):
    """The kernel's code by roles, from the first role's branch to the teardown; before them the role that is a function, if there is one."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(build_mod.CSRC, name)).read())
    begin = text.index("if (warp == kProducerWarp) {")
    gather = re.findall(r"auto gather_rows = \[&\].*?\n  \};", text[:begin], re.S)
    return gather + re.split(r"\n  \} else ", text[begin:text.index("tc_fence_before();\n  __syncthreads();", begin)])


# the roles of each kernel, and how many of them wait as whole warps
@pytest.mark.parametrize("name,n_roles,whole", [("gemm_pair.cu", 3, 3), ("gemm_stream.cu", 4, 4), ("gemm_tc.cu", 4, 3), ("step_ffn.cu", 5, 5)])
def test_no_lane_gives_up_by_itself(name, n_roles, whole):
    roles = _loops(name)
    assert len(roles) == n_roles
    assert sum("mbar_wait_warp(" in r for r in roles) >= whole
    for role in roles:
        if re.search(r"\bmbar_wait\(", role):  # every thread for itself, to the end of the role
            assert not re.search(WHOLE_WARP, role)
        # a wait by polling decides for the whole warp whether it goes on, and whether it gives up
        for poll in re.findall(r"for \(uint32_t polls = 0;[^{]*\{.*?\n {8,10}\}", role, re.S):
            assert "__all_sync" in poll.split("++polls")[0] and not re.search(r"if \((?!!__all_sync)[^)]*limit", poll)


def test_the_wait_for_a_counter_is_a_whole_warps():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(build_mod.CSRC, "step_ffn.cu")).read())
    body = re.search(r"bool wait_count\(.*?\n\}", text, re.S).group(0)
    assert re.findall(r"if \((.*)\) (?:break|return false);", body) == ["__all_sync(0xffffffffu, v >= want)",
                                                                      "!__all_sync(0xffffffffu, *abort_flag == 0 && now - t0 <= limit)"]
