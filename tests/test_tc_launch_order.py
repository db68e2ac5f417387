"""Source check (CPU only): a kernel that allocates tensor memory lets the next launch start only after
its allocation.

A CTA of the next launch holds its own tensor memory while it waits for this launch to end, so a CTA
that had allowed it earlier and still wanted tensor memory could wait for it without end."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_04896_gb300", "csrc")


def _kernels():
    """(file, text from one __global__ to the next) of every kernel that allocates tensor memory."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for body in text.split("__global__")[1:]:
            if "tcgen05.alloc" in body:
                yield os.path.basename(path), body


def test_dependents_start_after_the_allocation():
    found = list(_kernels())
    assert {f for f, _ in found} == {"croft_tc_kernel.cuh", "croft_tc_two_kernel.cuh"}
    for name, body in found:
        alloc = body.index("tcgen05.alloc")
        calls = [m.start() for m in re.finditer(r"pdl_allow_dependents\(\)|griddepcontrol\.launch_dependents", body)]
        assert all(c > alloc for c in calls), name
        # by the allocating warp: the call stands in the block that the allocation stands in
        for c in calls:
            assert body.rfind("if (tid < 32) {", 0, c) < alloc < c < body.index("}", alloc), name
