"""A pair's start, read in the source: no run can be relied on to show an order that is missing."""
import os
import re

KERNEL = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_24953_b200", "csrc", "gemm_blockscaled.cu")


def test_the_warp_that_allocates_tensor_memory_arrives_behind_its_allocation():
    # the leader's MMAs write the second CTA's tensor memory: every warp's start waits for both allocations
    code = re.sub(r"//[^\n]*", "", open(KERNEL).read())
    kernel = code[code.index("gemm_block_scaled_kernel("):]
    start = kernel[:kernel.index("wait_for_predecessor();")]
    allocation = start.index('"tcgen05.alloc.cta_group::2')
    early = re.findall(r"(if \([^\n]*\))[^;]*?cluster_arrive(?:_relaxed)?\(\);", start[:allocation])
    assert early == ["if (CTAS == 2)", "if (CTAS == 2 && warp != 1)"], early          # warp 4, and all others but warp 1
    assert "if (warp == 4)" in start[:start.index("if (CTAS == 2) cluster_arrive")]
    assert re.search(r"tcgen05_fence_before\(\);\s*cluster_arrive\(\);", start[allocation:])   # release
    assert start[allocation:].count("cluster_arrive") == 1
