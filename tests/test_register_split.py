"""Register split of the fused kernels (setmaxnreg): every warp of a warpgroup has to execute the same
instruction, so a kernel holds one decrease and one increase, each taken by whole warpgroups (asserted
where the warps' roles are defined)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1702_04728_gb300", "csrc")


@pytest.mark.parametrize("source", ["fused_fp32.cu", "fused_tc.cu"])
def test_one_setmaxnreg_of_each_kind_per_kernel(source):
    text = open(os.path.join(CSRC, source)).read()
    assert re.findall(r'"setmaxnreg\.(\w+)\.', text).count("dec") == 1
    assert re.findall(r'"setmaxnreg\.(\w+)\.', text).count("inc") == 1
