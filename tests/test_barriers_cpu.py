"""The group barrier as the source states it.  The two-codeword kernels read
shared memory by volatile asm without a memory clobber; such a read is ordered
after ordinary stores only by an asm statement that has the clobber, so every
barrier of a group, the one-warp form included, has to be one."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_05795_gb300", "csrc")


def test_group_barriers_are_asm_with_a_memory_clobber():
    text = open(os.path.join(CSRC, "decode_impl.cuh")).read()
    grp = re.sub(r"//[^\n]*", "", re.search(r"struct Grp \{.*?\n\};", text, re.S).group(0))
    asms = re.findall(r"asm volatile\((.*?)\);", grp, re.S)
    assert any("bar.warp.sync" in a for a in asms) and any("bar.sync" in a for a in asms)
    assert all('"memory"' in a for a in asms)
    assert "__syncwarp" not in grp  # (its reductions use the same barrier)
