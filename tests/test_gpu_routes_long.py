"""The default route by cache length: on either side of the lines in rows and keys (short caches: test_gpu_routes.py)."""
import pytest
import torch

from paper_2510_02329_b200 import binding, synth
from perf import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n,gamma,keys,persistent", [
    (synth.LLAMA_8B, 1, 8, 900, True), (synth.LLAMA_8B, 1, 8, 4096, True), (synth.LLAMA_8B, 1, 9, 900, False), (synth.LLAMA_8B, 1, 9, 500, True),
    (synth.LLAMA_8B, 1, 9, 503, False), (synth.LLAMA_8B, 2, 4, 900, True), (synth.LLAMA_8B, 2, 5, 900, False), (synth.LLAMA_8B, 3, 2, 900, False),
    (synth.LLAMA_8B, 4, 1, 900, True), (synth.QWEN_32B, 1, 8, 900, True), (synth.QWEN_32B, 1, 9, 900, False), (synth.QWEN_32B, 2, 4, 900, True),
    (synth.QWEN_32B, 2, 6, 900, False), (synth.QWEN_32B, 3, 3, 900, False),
    (synth.LLAMA_1B, 1, 14, 900, True), (synth.LLAMA_1B, 1, 15, 900, False), (synth.LLAMA_1B, 1, 15, 239, True), (synth.LLAMA_1B, 1, 15, 240, False),
    (synth.LLAMA_1B, 3, 3, 300, False), (synth.LLAMA_1B, 4, 1, 300, True)], ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_default_route_by_keys(shape, n, gamma, keys, persistent):
    """The step of either route gives the same results within the bf16 bounds."""
    target = cases.make_model(shape.cut(1, vocab=1000), torch.bfloat16, 3, 64)
    kv = cases.make_cache(target, [keys] * n, gamma + 2, 3)
    drafts = torch.randint(0, 1000, (n, gamma), dtype=torch.int32, device="cuda")
    got = []
    for step_impl in (2, 0 if persistent else 1):
        target.set_option("step_impl", step_impl)
        for name in ("graph", "timing"):
            target.set_option(name, int(name == "timing"))
        out = binding.VerifyBuffers(n, gamma, shape.d_model, 1000, debug=True)
        kv.set_pending(list(range(n)), [7 + b for b in range(n)])
        binding.verify(target, kv, list(range(n)), drafts, out, commit=False)
        target.sync()
        assert (target.kernel_time("verify_step")[1] > 0) == (persistent == (step_impl == 2))
        got.append(out)
    assert torch.allclose(got[0].dbg_logits, got[1].dbg_logits, atol=2e-2, rtol=2e-2)
    assert torch.allclose(got[0].judge_scores, got[1].judge_scores, atol=1e-3)
    kv.close()
    target.close()
