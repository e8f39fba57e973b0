"""Kernels that entry points launch as programmatic dependents of whatever the caller's stream holds.  The kernel in front may be anybody's: it
may signal its dependents early and allocate tensor memory afterwards, and a dependent that already holds the columns while it waits for that
kernel to complete would keep both waiting for good.  So nothing is taken before the wait (read in the source: the case itself is not run)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_00150_b200", "csrc")
KERNEL = re.compile(r"__global__ void __launch_bounds__\([^;{]*?\)\s*(\w+)\(")


def kernel_bodies(name):
    text = open(os.path.join(CSRC, name)).read()
    at = [(m.group(1), m.start()) for m in KERNEL.finditer(text)] + [(None, len(text))]
    return {k: re.sub(r"//[^\n]*", "", text[a:b]) for (k, a), (_, b) in zip(at, at[1:])}


@pytest.mark.parametrize("source,kernel,from_entry", [
    ("amq_bgemm_resident.cu", "bgemm_resident_kernel", "!a.early_weights"),
    ("amq_bgemm_tc.cu", "bgemm_tc_kernel", "a.from_entry"),
    ("amq_bgemm_tc.cu", "bgemm_tc_persistent_kernel", "a.from_entry"),
])
def test_products_of_an_entry_point_take_tensor_memory_after_the_wait(source, kernel, from_entry):
    body = kernel_bodies(source)[kernel]
    before, alloc, after = body.partition('asm volatile("tcgen05.alloc')
    assert alloc, "the allocation is not where this test looks for it"
    branch = before[before.rindex("{"):]                    # the allocating warp's branch, up to the allocation
    assert "if (%s) grid_dependency_wait();" % from_entry in branch
    # no bounded wait runs beside the kernel in front either: the whole CTA meets behind that warp first
    assert "mbar_wait" not in before and after.index("__syncthreads()") < after.index("mbar_wait" if "mbar_wait" in after else "res_feed")
