"""Prefill in wide blocks: the edges of its blocks, on an empty and on a ragged non-empty cache, against the oracle."""
import numpy as np
import pytest
import torch

import harness
import helpers
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth
from test_gpu_extensions import _empty_case

pytestmark = pytest.mark.gpu

HD128 = synth.ModelShape("hd128-gqa", 2, 256, 4, 2, 128, 512, 1000, rope_theta=5e5, qkv_bias=True)
HD128_G4 = synth.ModelShape("hd128-group4", 2, 512, 4, 1, 128, 256, 640)


@pytest.mark.parametrize("shape", [synth.TINY, HD128, HD128_G4], ids=lambda s: s.name)
@pytest.mark.parametrize("before,n", [(0, 33), (0, 64), (7, 512), (21, 513), (0, 1025)])
def test_wide_prefill(shape, before, n):
    """One block, a full one, a full and a tiny one, three; `before` tokens in the cache already (a page's middle)."""
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


def _verify(case, si, shape):
    from paper_2510_02329_b200 import binding as b
    out = b.VerifyBuffers(1, 3, shape.d_model, shape.vocab, debug=True)
    b.verify(case.target, case.kv, [0], torch.from_numpy(si.draft_ids).cuda(), out, commit=False)
    case.target.sync()
    return out.dbg_logits.cpu().numpy()[0]
