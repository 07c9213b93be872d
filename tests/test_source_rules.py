"""Rules of the device code that no run can show: a branch on a kernel's abort flag, which another
warp sets at any moment, must be taken by whole warps (shuffles and tensor-memory loads follow)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_10557_gb300", "csrc")


@pytest.mark.parametrize("name", ["tc_filter.cu", "tc_dgemm.cu"])
def test_abort_flag_is_read_by_whole_warps(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    reads = [m.start() for m in re.finditer(r"\*abort_sh\b(?!\s*=[^=])", text)]
    lone = []
    for i in reads:
        line = text[text.rfind("\n", 0, i) + 1:text.find("\n", i)]
        if "volatile int*" in line or "__all_sync(0xffffffffu, *abort_sh == 0)" in line:
            continue
        if "threadIdx.x == 0 && *abort_sh" in line:  # one thread, after the block barrier of the teardown
            continue
        lone.append(line.strip())
    assert len(reads) >= 2 and lone == []
