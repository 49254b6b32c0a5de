"""Waits of the kernels for the kernel in front of them, read from the sources (a missing fence shows in no result that can be relied on)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_12023_b200", "csrc")
COPY = re.compile(r"\b(tma_load_2d|bulk_load|issue_box|issue_codes)\(")


def test_copies_behind_a_wait_are_behind_its_proxy_fence():
    """What the kernel in front wrote with ordinary stores is read by TMA and bulk copies through the async proxy: a thread that requests them
    behind griddepcontrol.wait passes fence.proxy.async first (pdl_wait_for_copies).  The plain wait is for roles that read with loads: nothing
    that follows it, up to the next role or the next barrier of the block, requests a copy."""
    files = {f: open(os.path.join(CSRC, f)).read() for f in ("linear_swap.cuh", "linear_tc.cuh", "linear_tc2.cuh", "lora_grad.cuh")}
    for f, text in files.items():
        assert "pdl_wait_for_copies()" in text, f
        for after in text.split("pdl_wait();")[1:]:
            role = re.split(r"\} else if \(warp|__syncthreads\(\)", after)[0]
            assert not COPY.search(role), f"{f}: copy requested behind a wait without the fence: {role[:200]}"
    body = files["linear_tc.cuh"].split("void lowrank_body(")[1].split("template <bool BWD>")[0]
    assert "pdl_wait_for_copies()" in body and "pdl_wait();" not in body            # its copies stand behind a barrier of the block
