"""Prefill in wide blocks: the edges of its blocks, on an empty and on a ragged non-empty cache, against the oracle."""
import numpy as np
import pytest
import torch

import harness
import helpers
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import binding, synth
from perf import cases
from test_gpu_extensions import _empty_case

pytestmark = pytest.mark.gpu

HD128 = synth.ModelShape("hd128-gqa", 2, 256, 4, 2, 128, 512, 1000, rope_theta=5e5, qkv_bias=True)
HD128_G4 = synth.ModelShape("hd128-group4", 2, 512, 4, 1, 128, 256, 640)


@pytest.mark.parametrize("shape", [synth.TINY, HD128, HD128_G4], ids=lambda s: s.name)
@pytest.mark.parametrize("before,n", [(0, 33), (0, 64), (7, 512), (21, 513), (0, 1025)])
def test_wide_prefill(shape, before, n):
    """One block, one of 512 rows (entries of 32; two of 264 where they are 24), a token more (two blocks of equal size), three blocks;
    `before` tokens in the cache already (a page's middle)."""
    case = _empty_case(shape, torch.bfloat16, room=1100)
    try:
        prompt = synth.token_ids(shape.vocab, before + n, seed=51, stream=9)
        if before:
            case.kv.prefill(0, prompt[:before], want_next=False)
        nxt = case.kv.prefill(0, prompt[before:])
        assert case.kv.lengths([0]) == [before + n]
        bf, cache = orc.prefill(case.osh, case.top64, case.model.layer64, prompt)
        tol = harness.tol_for(torch.bfloat16, float(np.abs(bf.logits).max()))
        for l in range(shape.n_layers):
            k, v = case.kv.read(0, l, 0, before + n)
            for got, want in ((k, cache[l][0]), (v, cache[l][1])):
                err = np.abs(got.cpu().double().numpy() - want)
                assert (err <= tol.delta(want)).all(), (l, err.max())
        last = bf.logits[-1]
        assert nxt == int(np.argmax(last)) or last.max() - last[nxt] <= 2 * tol.delta(np.abs(last).max())
        # the pending token and the length are those the next step starts from
        si = synth.step_inputs(shape.vocab, 1, 3, seed=52)
        out = _verify(case, si, shape)
        stored = [tuple(helpers.np64(t) for t in case.kv.read(0, l, 0, before + n)) for l in range(shape.n_layers)]
        _, f = orc.verify(case.osh, case.top64, case.model.layer64, [nxt], si.draft_ids, [stored], mode=orc.GREEDY,
                          judge_w=case.judge_w64, theta=0.5)
        assert (np.abs(out - f[0].logits) <= tol.delta(f[0].logits)).all()
    finally:
        case.close()


@pytest.mark.parametrize("shape,n,block", [(synth.LLAMA_8B.cut(2, vocab=2048), 1000, 504), (synth.LLAMA_1B.cut(2, vocab=2048), 700, 360)],
                         ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_a_long_prompt_leaves_the_bits_of_its_blocks(shape, n, block):
    """At most 512 rows go through the layers at once, in blocks of equal size: the same calls by hand leave the same cache."""
    target = cases.make_model(shape, torch.bfloat16, 53, 64)
    kv = binding.KVCache(target, 1, n // 16 + 2)
    prompt = synth.token_ids(shape.vocab, n, seed=53, stream=9).tolist()
    stored = []
    for piece in (n, block):
        kv.rollback([0], [0])
        for i in range(0, n, piece):
            kv.prefill(0, prompt[i:i + piece], want_next=False)
        stored.append([kv.read(0, l, 0, n) for l in range(shape.n_layers)])
    for whole, parts in zip(*stored):
        assert torch.equal(whole[0], parts[0]) and torch.equal(whole[1], parts[1])
    kv.close()
    target.close()


def _verify(case, si, shape):
    out = binding.VerifyBuffers(1, 3, shape.d_model, shape.vocab, debug=True)
    binding.verify(case.target, case.kv, [0], torch.from_numpy(si.draft_ids).cuda(), out, commit=False)
    case.target.sync()
    return out.dbg_logits.cpu().numpy()[0]
