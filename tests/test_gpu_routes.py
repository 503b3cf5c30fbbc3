"""Which steps run as one persistent launch by default: on either side of the lines by widths, sequences and rows."""
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu

D512 = synth.ModelShape("d512", 1, 512, 8, 8, 64, 2048, 1000)
D1536 = synth.ModelShape("d1536", 1, 1536, 24, 6, 64, 6144, 1000)
HD128, HD64 = synth.LLAMA_8B.cut(1, vocab=1000), synth.LLAMA_1B.cut(1, vocab=1000)


@pytest.mark.parametrize("shape,n,gamma,persistent", [
    (D512, 1, 8, False), (D1536, 1, 8, True),
    (HD128, 1, 16, True), (HD128, 1, 17, False), (HD128, 2, 5, True), (HD128, 2, 6, False), (HD128, 6, 1, True), (HD128, 5, 2, False),
    (HD64, 1, 23, True), (HD64, 4, 5, True), (HD64, 4, 6, False), (HD64, 6, 1, True), (HD64, 8, 1, False)],
    ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_default_route(shape, n, gamma, persistent):
    case = harness.Case(shape, torch.bfloat16, [30 + 11 * b for b in range(n)], gamma, seed=27, cache="fill", gen_device="cuda").gpu_setup()
    try:
        for name in ("graph", "timing"):
            case.target.set_option(name, int(name == "timing"))
        v, f = case.run_oracle(orc.GREEDY)
        rep = harness.compare(case, v, f, case.run_gpu(orc.GREEDY), orc.GREEDY)
        assert rep.exact + rep.margin == n
        assert (case.target.kernel_time("verify_step")[1] > 0) == persistent
    finally:
        case.close()
