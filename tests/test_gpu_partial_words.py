"""The persistent kernel's exchange of partial sums: words of three rows and a tag, of which the last of a group may carry one
row only.  Step after step on the same inputs, at the row counts around the kernel's instantiations (up to 8, 12, 48 rows)."""
import numpy as np
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,gamma", [(1, 1), (1, 3), (1, 5), (1, 6), (1, 7), (4, 1), (1, 8), (2, 4), (1, 11), (1, 12), (3, 15)],
                         ids=lambda x: str(x))
@pytest.mark.parametrize("shape", [synth.LLAMA_8B.cut(2, vocab=2048), synth.LLAMA_1B.cut(2, vocab=2048)], ids=lambda s: s.name)
def test_steps_repeat(shape, n, gamma):
    case = harness.Case(shape, torch.bfloat16, [200 - 30 * b for b in range(n)], gamma, seed=16, cache="fill", gen_device="cuda").gpu_setup()
    try:
        case.target.set_option("step_impl", 1)
        v, f = case.run_oracle(orc.GREEDY)
        runs = [case.run_gpu(orc.GREEDY) for _ in range(8)]
        rep = harness.compare(case, v, f, runs[0], orc.GREEDY)
        assert rep.exact + rep.margin == n
        assert rep.max_hidden_err < 2e-3, rep      # what the two activation planes leave elsewhere in these tests
        for again in runs[1:]:
            np.testing.assert_array_equal(again["hidden"], runs[0]["hidden"])
    finally:
        case.close()
