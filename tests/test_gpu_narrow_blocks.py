"""Steps of at most 16 rows on the per-stage path: their row blocks are halved between the epilogue's two groups (8 rows each);
17 rows are the first of the wider blocks."""
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu

SPLIT = synth.ModelShape("narrow-split", 2, 1152, 8, 2, 128, 4160, 1920, qkv_bias=True)      # odd tiles; K shared by several pairs
HD64 = synth.ModelShape("narrow-hd64", 2, 512, 8, 4, 64, 1024, 1000)                         # vocabulary ends inside a tile


@pytest.mark.parametrize("shape", [SPLIT, HD64], ids=lambda s: s.name)
@pytest.mark.parametrize("n,gamma", [(1, 1), (1, 6), (1, 7), (1, 8), (3, 4), (1, 15), (2, 7), (1, 16)])
def test_narrow_row_blocks(shape, n, gamma):
    case = harness.Case(shape, torch.bfloat16, [40 + 37 * b for b in range(n)], gamma, seed=23, cache="fill").gpu_setup(max_rows=n * (gamma + 1))
    try:
        case.target.set_option("step_impl", 0)
        for mode in (orc.GREEDY, orc.SAMPLING):
            v, f = case.run_oracle(mode)
            rep = harness.compare(case, v, f, case.run_gpu(mode), mode)
            assert rep.exact + rep.margin == n
            assert rep.max_hidden_err < 2e-3, rep   # what the two activation planes leave elsewhere in these tests
    finally:
        case.close()
