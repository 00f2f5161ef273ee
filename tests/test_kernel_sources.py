"""Rules of the kernel sources that no input can show without a failed wait or
a second device, checked on the text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1308_2864_gb300", "csrc")


def read(name):
    return open(os.path.join(CSRC, name), encoding="utf-8").read()


def test_wide_update_warps_leave_their_waits_by_vote():
    # lanes of a warp may see the abort flag at different polls; a warp-wide
    # instruction (warp barrier, tensor-memory load) behind such a wait needs all
    # of them, so the loading warps leave or stay by vote
    k = read("ks_tc.cu").split("combine_tcw_kernel(\n", 1)[1]
    warps = k.split("if (warp < 8) {", 1)[1].split("} else if (warp == 8 && lane == 0) {", 1)[0]
    waits = re.findall(r"const bool (\w+) =[^;]*role_wait\(", warps)
    assert len(waits) == warps.count("role_wait(") == 2
    for name in waits:
        assert re.search(r"__all_sync\(0xffffffffu, %s\)" % name, warps)
