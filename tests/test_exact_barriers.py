"""The token-by-token fp32 kernel's aligned barriers (csrc/wkv6_exact.cuh), read in its source: a whole warp has to execute one at
once, so where lanes may have parted before it the warp meets first."""
import os
import re

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_12077_b200", "csrc", "wkv6_exact.cuh")).read()
KERNEL = SRC[SRC.index("wkv6_exact_kernel(const IO*"):SRC.index("inline cudaError_t launch_exact_as")]
ALIGNED = r'asm volatile\("[^;]*?(bar\.sync|\.aligned)'


def meets_first(text, at):
    return text[:at].rstrip().endswith("__syncwarp();")


def test_a_warp_meets_before_an_aligned_barrier():
    barriers = [m.start() for m in re.finditer(ALIGNED, KERNEL)]
    assert all(meets_first(KERNEL, at) for at in barriers), [KERNEL[at - 80:at + 60] for at in barriers if not meets_first(KERNEL, at)]
    for name in ("ex_bar_sync", "ex_bar_or"):
        assert KERNEL.count(name + "(") >= 1
        assert re.search(name + r"\([^)]*\)\n\{\n    __syncwarp\(\);\n    asm", SRC)
    for m in re.finditer(r"(if \(G > 1\) )cluster_(wait|arrive)\(\)", KERNEL):
        assert meets_first(KERNEL, m.start())


def test_a_warp_meets_after_a_wait_that_each_lane_ends_by_itself():
    waits = re.findall(r"cluster_mbar_wait\([^;]*;\s*(\S+)", KERNEL)
    assert len(waits) == 2 and set(waits) == {"__syncwarp();"}
