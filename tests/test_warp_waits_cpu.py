"""A bounded wait that runs out must be answered alike by all lanes of a warp wherever the code behind it is the whole warp's
(tensor-memory loads, stmatrix, __syncwarp): a lane that left by itself would be waited for without a limit.  Read from the
sources, because a run that shows it would hang."""
import os
import re

import pytest

from paper_2609_00993_b200 import build as build_mod

# what a whole warp executes together
WHOLE_WARP = r"__syncwarp|__shfl|__all_sync|__ballot|elect_one|tmem_ld|stmatrix|mbar_wait_warp"


def _loops(name):
    """The kernel's code by roles, from the first role's branch to the teardown."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(build_mod.CSRC, name)).read())
    begin = text.index("if (warp == kProducerWarp) {")
    return re.split(r"\n  \} else ", text[begin:text.index("tc_fence_before();\n  __syncthreads();", begin)])


@pytest.mark.parametrize("name", ["gemm_pair.cu", "gemm_stream.cu", "gemm_tc.cu"])
def test_no_lane_gives_up_by_itself(name):
    roles = _loops(name)
    assert len(roles) == (4 if name == "gemm_tc.cu" else 3)
    assert sum("mbar_wait_warp(" in r for r in roles) >= 3
    for role in roles:
        if re.search(r"\bmbar_wait\(", role):  # every thread for itself, to the end of the role
            assert not re.search(WHOLE_WARP, role)
