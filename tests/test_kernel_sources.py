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


def test_function_attributes_are_not_set_once_per_process():
    # a kernel's shared-memory limit belongs to a device: set on the first launch
    # of a process only, a launch on a second device lacks it.  Every call of
    # cudaFuncSetAttribute belongs to a function that problem or batch creation runs
    setters = {"configure_", "stencil_opt_in", "batch_cg_setup", "cg_grid_blocks"}
    for f in sorted(os.listdir(CSRC)):
        src = read(f)
        if "cudaFuncSetAttribute" not in src:
            continue
        assert not re.search(r"call_once\([^;]*cudaFuncSetAttribute", src, re.S), f
        for m in re.finditer(r"cudaFuncSetAttribute\(", src):
            head = re.findall(r"^(?:static )?(?:inline )?[\w: ]+ \**(\w+)\([^;{]*\) \{", src[:m.start()],
                              re.M)
            assert any(head[-1].startswith(s) for s in setters), (f, head[-1])
