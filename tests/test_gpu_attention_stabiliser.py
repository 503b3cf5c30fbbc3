"""The tcgen05 attention's stabiliser: caches whose later keys score far above the earlier ones, so that the running
maximum has to move in the middle of a segment and what was accumulated is rescaled.  Several segments per block, one and two
query chunks per group, against the oracle."""
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu

HD128 = synth.ModelShape("hd128-group4", 2, 512, 8, 2, 128, 1024, 2048)


@pytest.mark.parametrize("lens,gamma", [([900, 2100, 300, 129, 700, 1500, 40], 7), ([900, 2100, 300], 7), ([1300, 400], 20)],
                         ids=["7", "3", "84-query-rows"])
def test_scores_that_outgrow_the_stabiliser(lens, gamma):
    case = harness.Case(HD128, torch.bfloat16, lens, gamma, seed=12, cache="fill")
    for seq in case.cache_t:
        for layer, (k, v) in enumerate(seq):
            k = k.float()
            for at, factor in ((128, 4.0), (384, 10.0), (640, 0.5), (1000, 20.0)):     # growing, shrinking, growing again
                k[at:] = k[at:] * factor if at != 640 else k[at:] * 0.5
            seq[layer] = (k.to(torch.bfloat16), v)
    case.gpu_setup(max_rows=len(lens) * (gamma + 1))
    try:
        for name, value in (("step_impl", 0), ("attn_impl", 2)):
            case.target.set_option(name, value)
        v, f = case.run_oracle(orc.GREEDY)
        rep = harness.compare(case, v, f, case.run_gpu(orc.GREEDY), orc.GREEDY)
        assert rep.exact + rep.margin == len(lens)
    finally:
        case.close()
