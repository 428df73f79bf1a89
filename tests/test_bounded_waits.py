"""A CTA whose wait has run out may have copies in flight into its shared memory: it pauses before it
leaves.  No wait is made to run out on a device here; the sources say whether a kernel that waits pauses."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_09708_b200", "csrc")
KERNELS = [p for p in sorted(glob.glob(os.path.join(CSRC, "*.cu"))) if "tma_load" in open(p).read()]


def kernel_bodies(text):
    for m in re.finditer(r"^(?:template <[^>]*>\n)?__global__ .*?^\{$(.*?)^\}$", text, re.S | re.M):
        yield m.group(1)


@pytest.mark.parametrize("path", KERNELS, ids=os.path.basename)
def test_a_kernel_that_loads_pauses_before_it_leaves(path):
    bodies = [b for b in kernel_bodies(open(path).read()) if "tma_load" in b]
    assert bodies
    for body in bodies:
        at_the_end = r"if \(\*abort_flag\).*__nanosleep\(|if \(!ok\) let_copies_land\(\);\s*(tc_fence_before\(\);\s*)?__syncthreads\(\);"
        waits = [line for line in re.findall(r"[^\n]*mbar_wait\([^\n]*\n[^\n]*", body)]
        after_each = waits and all("let_copies_land()" in w for w in waits)
        assert after_each or re.search(at_the_end, body[max(body.rfind("mbar_wait("), 0):], re.S)
