"""How a CTA of a paired projection leaves its cluster, read from the kernel's source: nothing that may still be on its way to a
CTA outlives it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_02329_b200", "csrc")
SRC = open(os.path.join(CSRC, "sj_gemm_pair.cuh")).read()


def body(src, head):
    """The braces that follow `head`."""
    at = src.index("{", src.index(head))
    depth = 0
    for i in range(at, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[at:i]


def test_a_wait_that_runs_out_delays_its_warp_before_the_report():
    """The delay in which copies land is the expired wait's own, so it precedes the warp's report to the last cluster barrier
    wherever that is; behind a report it would hold its own CTA only."""
    wait = body(open(os.path.join(CSRC, "sj_gemm_tc.cuh")).read(), "bool mbar_wait(")
    assert 0 < wait.find("atomicCAS(status, DEV_OK, DEV_TIMEOUT)") < wait.find("__nanosleep(20000)")
    kernel = body(SRC, "k_gemm_pair(const __grid_constant__")
    assert "__nanosleep" not in kernel and not re.search(r"att_mbar_wait|(?<!mbar_)try_wait\(smem_u32\(&ctl->(?!xch)", kernel)
    assert kernel.count("cluster_arrive_all()") == 2                    # the epilogue's warps, the others
