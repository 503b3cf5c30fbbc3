"""fp32 models against the oracle, where their kernels' tiles end: row passes (4, 8 or 12 rows at a time), K and N that are no
multiples of a step or a tile, more and fewer units than blocks, caches that end inside, at and after a tile of keys."""
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu

SMALL = synth.ModelShape("small-f32", 2, 72, 4, 2, 64, 200, 777, qkv_bias=True)
WIDE = synth.ModelShape("wide-f32", 2, 1160, 6, 2, 128, 3000, 10501)


@pytest.mark.parametrize("shape,lens,gamma", [
    (SMALL, [0], 1), (SMALL, [1, 63], 1), (SMALL, [64, 65, 130], 3), (SMALL, [500], 12), (SMALL, [200, 3, 64, 129], 9),
    (WIDE, [64], 2), (WIDE, [333, 31], 4), (WIDE, [700, 0, 65], 7), (WIDE, [95], 30)], ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_against_the_oracle(shape, lens, gamma):
    case = harness.Case(shape, torch.float32, lens, gamma, seed=31, cache="fill").gpu_setup()
    try:
        for mode in (orc.GREEDY, orc.SAMPLING):
            v, f = case.run_oracle(mode)
            rep = harness.compare(case, v, f, case.run_gpu(mode), mode)
            assert rep.exact + rep.margin == len(lens)
            assert rep.max_hidden_err < 2e-5, rep   # sums of 3000 fp32 products, two layers: the library's fp32 cases state this
    finally:
        case.close()
