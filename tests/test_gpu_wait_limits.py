"""How long the library's bounded waits last before they give up: a second or so each, at the time that a poll takes here."""
import os
import re
import time

import pytest
import torch

import harness
from paper_2510_02329_b200 import binding, synth

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_02329_b200", "csrc")


def polls(name):
    """A limit as the kernels' sources state it; a name stands for another limit."""
    for f in ("sj_gemm_tc.cuh", "sj_gemm_pair.cuh", "sj_attn_tc.cuh", "sj_mega.cuh"):
        m = re.search(rf"constexpr uint32_t {name} = (?:1u << (\d+)|(\w+));", open(os.path.join(CSRC, f)).read())
        if m:
            return 1 << int(m.group(1)) if m.group(1) else polls(m.group(2))


@pytest.mark.parametrize("kind,names", [(0, ("kSpinLimit", "kPairSpin")), (1, ("kAttSpin",)), (2, ("kMegaSpin",))])
def test_a_wait_gives_up_after_a_second_or_so(kind, names):
    """A drill of 2^14 polls, behind the first 2^13 whose pauses are shorter, gives the time of one."""
    target = harness.Case(synth.TINY, torch.bfloat16, [20], 1, seed=0).gpu_setup().target
    took = []
    for n in (1 << 13, 1 << 13, (1 << 13) + (1 << 14)):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        target.expire_wait(kind, n)
        with pytest.raises(binding.SjError):
            target.sync()
        took.append(time.perf_counter() - t0)
    poll = (took[2] - took[1]) / (1 << 14)
    for name in names:
        assert 0.3 < poll * polls(name) < 3, (name, polls(name), poll)
