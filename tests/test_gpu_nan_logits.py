"""Logits that are all NaN (a broken checkpoint): the emitted token is still one of the vocabulary, token 0."""
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,options", [(torch.bfloat16, {"step_impl": 1}), (torch.bfloat16, {"step_impl": 0}), (torch.bfloat16, {"gemm_impl": 0}),
                                           (torch.float32, {})], ids=["persistent", "per-stage", "cudacore", "f32"])
def test_nan_logits(dtype, options):
    case = harness.Case(synth.TINY, dtype, [20, 33], 4, seed=25, cache="fill")
    case.model.top["lm_head"][:] = float("nan")
    case.gpu_setup()
    try:
        for k, v in options.items():
            case.target.set_option(k, v)
        g = case.run_gpu(orc.GREEDY, use_judge=False)
        assert (g["accepted_len"] == 0).all() and (g["next_token"] == 0).all(), g["next_token"]
    finally:
        case.close()
