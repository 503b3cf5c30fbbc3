"""The [rows, vocabulary] logits of sampling are memory of the targets that sample."""
import numpy as np
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu

WIDE_VOCAB = synth.ModelShape("wide-vocab", 1, 256, 4, 4, 64, 256, 128256)


def _held():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    return total - free - torch.cuda.memory_reserved()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
def test_only_sampling_targets_hold_logits(dtype):
    case = harness.Case(WIDE_VOCAB, dtype, [40, 7, 100], 4, seed=23, cache="fill")
    before = _held()
    case.gpu_setup(max_rows=512)
    try:
        all_rows = 512 * WIDE_VOCAB.vocab * 4
        created = _held() - before
        assert created < all_rows // 2, created                     # 263 MB of logits would be most of it
        for mode in (orc.GREEDY, orc.SAMPLING):
            v, f = case.run_oracle(mode)
            rep = harness.compare(case, v, f, case.run_gpu(mode), mode)
            assert rep.exact + rep.margin == 3
            grown = _held() - before - created
            assert grown < all_rows // 2, grown                     # the 15 rows that sample; the kernels' own code is 96 MB of it
    finally:
        case.close()


def test_more_rows_after_fewer_in_sampling():
    """The buffer grows with the rows: 5, then 15, then 5 again, captured steps included."""
    case = harness.Case(synth.LLAMA_8B.cut(1, vocab=40000), torch.bfloat16, [40, 7, 100], 4, seed=24, cache="fill", gen_device="cuda").gpu_setup()
    try:
        from paper_2510_02329_b200 import binding
        for impl in (0, 1):
            case.target.set_option("step_impl", impl)
            tokens = []
            for n in (1, 3, 1, 3):
                out = binding.VerifyBuffers(n, 4)
                case.kv.set_pending(list(range(n)), case.inputs.pending[:n])
                binding.verify(case.target, case.kv, list(range(n)), case.d_draft[:n].contiguous(), out, mode=binding.MODE_SAMPLING,
                               draft_q_tok=case.d_qtok[:n].contiguous(), draft_q_full=case.d_qfull[:n].contiguous(),
                               uniforms=case.d_unif[:n].contiguous(), use_judge=False, commit=False)
                case.target.sync()
                tokens.append(out.next_token.cpu().numpy())
            assert tokens[0] == tokens[2] and (tokens[1] == tokens[3]).all() and tokens[0][0] == tokens[1][0]
            v, _ = case.run_oracle(orc.SAMPLING, use_judge=False)
            np.testing.assert_array_equal(tokens[3], [x.next_token for x in v])
    finally:
        case.close()
