"""Rules of the device code that no run on a GPU can show to be kept."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_16536_b200", "csrc")


def _kernels(text):
    """(name, body) of every __global__ function, comments removed."""
    text = re.sub(r"__launch_bounds__\([^)]*\)", "", re.sub(r"//[^\n]*", "", text))
    for m in re.finditer(r"__global__[^{;]*?(\w+)\s*\(", text):
        start = text.index("{", text.index(")", m.end()))
        depth = 0
        for i in range(start, len(text)):
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            if depth == 0:
                yield m.group(1), text[start:i + 1]
                break


def test_kernels_that_let_the_next_launch_start_wait_for_the_one_in_front_before_they_return():
    """A kernel that triggers the next launch early is what that launch waits for: if it could end without its own wait,
    the next kernel would run beside the one in front of it."""
    seen = []
    for name, body in _kernels(open(os.path.join(CSRC, "kernels_basic.cuh")).read()):
        body = body.replace("next_launch_may_start()", "griddepcontrol.launch_dependents").replace("wait_for_launch_before()", "griddepcontrol.wait")
        if "griddepcontrol.launch_dependents" in body:
            seen.append(name)
            assert not re.search(r"\breturn\b", body[:body.index("griddepcontrol.wait")]), name
    assert sorted(seen) == ["dequant_kernel", "pack_kernel", "quantize_kernel", "stage_activations_kernel", "tile_splitk_reduce_kernel"]


def test_a_barrier_tested_without_waiting_steers_a_warp_only_by_vote():
    """Each lane gets its own answer from a test of a barrier that other warps complete meanwhile.  What comes behind it is
    for the whole warp (elect.sync, __syncwarp, which MMAs go out), so that the lanes have to agree first."""
    uses = 0
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for m in re.finditer(r"(\S*\s*\S*)\bmbar_test\(", text):
            if "bool" in m.group(1):                     # the definition
                continue
            uses += 1
            assert re.search(r"__(all|any)_sync\(0xffffffffu,\s*$", m.group(1)), (name, m.group(0))
    assert uses == 1
