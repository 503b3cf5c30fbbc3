"""Kernels that take tensor memory let their dependents start only when they have it, read from the sources: allocation waits
until enough is free, and a dependent on the same SM would hold its share until this kernel has ended."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_02329_b200", "csrc")


def kernels():
    """(file, name, body) of every kernel that allocates tensor memory."""
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^)]*\)\s*)?(k_\w+)\(", src):
            at, depth = src.index("{", m.end()), 0
            for i in range(at, len(src)):
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                if depth == 0:
                    break
            if "tcgen05.alloc" in src[at:i]:
                yield f, m.group(1), src[at:i]


@pytest.mark.parametrize("f,name,body", list(kernels()), ids=lambda x: x if x.startswith("k_") else "")
def test_tensor_memory_comes_before_the_dependents(f, name, body):
    launch = body.find("pdl_launch()")
    assert launch < 0 or body.index("tcgen05.alloc") < body.index("__syncthreads()", body.index("tcgen05.alloc")) < launch


def test_the_kernels_are_found():
    assert {"k_attn_t5", "k_gemm_pair", "k_gemm_tc"} <= {name for _, name, _ in kernels()}
