"""Pending tokens, page numbers, lengths and roll-backs of many sequences at once: each travels as the parameters of one
kernel, up to the largest batch.  A sequence named twice in one call ends as if its entries came one after another."""
import random

import pytest
import torch

import harness
from paper_2510_02329_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,step_impl", [(1, 0), (1, 1), (24, 1), (255, 0), (256, 0)])
def test_a_large_batch_equals_its_parts(B, step_impl):
    """Every sequence needs a new page (16 cached tokens) in the step; parts of at most 8 sequences are the reference."""
    c = harness.Case(synth.TINY, torch.bfloat16, [16], 1, seed=5, cache="fill").gpu_setup(max_rows=512)
    c.target.set_option("step_impl", step_impl)
    shape, ids = synth.TINY, list(range(B))[::-1]
    g = torch.Generator().manual_seed(7)
    pending = torch.randint(0, shape.vocab, (B,), generator=g).tolist()
    drafts = torch.randint(0, shape.vocab, (B, 1), generator=g, dtype=torch.int32).cuda()

    def run(parts):
        kv = binding.KVCache(c.target, B, 2 * B + 4)
        for s in range(B):
            for l, (k, v) in enumerate(c.cache_t[0]):
                kv.fill(s, l, 0, k.cuda(), v.cuda())
        kv.set_len(ids, [16] * B)
        kv.set_pending(ids, pending)
        got = []
        for at in range(0, B, parts):
            out = binding.VerifyBuffers(min(parts, B - at), 1, shape.d_model, shape.vocab, debug=True)
            binding.verify(c.target, kv, ids[at:at + parts], drafts[at:at + parts].contiguous(), out, theta=0.5)
            got.append(out)
        c.target.sync()
        lens = kv.lengths(ids)
        to = [15 + i % 2 for i in range(B)]
        kv.rollback(ids, to)
        c.target.sync()
        assert kv.lengths(ids) == to
        kv.close()
        out = {n: torch.cat([getattr(o, n) for o in got]) for n in ("accepted_len", "next_token", "new_kv_len", "judge_scores", "dbg_logits")}
        assert lens == out["new_kv_len"].tolist() == (17 + out["accepted_len"]).tolist()
        return out

    whole, parts = run(B), run(8)
    # parts of another size run other kernels, whose sums differ in the last bits: the bounds of the bf16 paths
    assert torch.allclose(whole["dbg_logits"], parts["dbg_logits"], atol=2e-2, rtol=2e-2)
    assert torch.allclose(whole["judge_scores"], parts["judge_scores"], atol=1e-3)
    best = parts["dbg_logits"].topk(2, dim=2).values
    clear = ((best[:, :, 0] - best[:, :, 1]).min(dim=1).values > 4e-2) & ((parts["judge_scores"][:, 0] - 0.5).abs() > 2e-3)
    assert clear.sum() >= B // 4
    for n in ("accepted_len", "next_token"):
        assert torch.equal(whole[n][clear], parts[n][clear])
    c.close()


@pytest.mark.parametrize("n_seqs", [1, 5, 40])
def test_a_sequence_named_twice_ends_with_its_last_entry(n_seqs):
    """The largest batch of entries over a few sequences; roll-backs end at the shortest, the host's page count with them."""
    room, shape, ids = 96, synth.TINY, list(range(n_seqs))
    c = harness.Case(shape, torch.bfloat16, [16], 2, seed=5, cache="fill").gpu_setup(max_rows=256)
    kv = binding.KVCache(c.target, n_seqs, n_seqs * (room // 16) + 8)
    rows = torch.randn(room, shape.n_kv_heads, shape.head_dim, device="cuda").bfloat16()
    for s in ids:
        for l in range(shape.n_layers):
            kv.fill(s, l, 0, rows, rows)
    r = random.Random(n_seqs)
    drafts = torch.randint(0, shape.vocab, (n_seqs, 2), dtype=torch.int32, device="cuda")

    def logits():
        out = binding.VerifyBuffers(n_seqs, 2, shape.d_model, shape.vocab, debug=True)
        binding.verify(c.target, kv, ids, drafts, out, commit=False)
        c.target.sync()
        return out.dbg_logits

    for _ in range(20):
        named = ids + [r.randrange(n_seqs) for _ in range(256 - n_seqs)]
        r.shuffle(named)
        lens, tokens = [r.randrange(1, room - 3) for _ in named], [r.randrange(shape.vocab) for _ in named]
        last = dict(zip(named, zip(lens, tokens)))
        kv.set_len(named, lens)
        kv.set_pending(named, tokens)
        assert kv.lengths(ids) == [last[s][0] for s in ids]
        got = logits()
        kv.set_pending(ids, [last[s][1] for s in ids])
        assert torch.equal(got, logits())
        for s in ids:      # lengths() has given the pages beyond a sequence's length back
            kv.fill(s, 0, 0, rows, rows)
        kv.set_len(ids, [room] * n_seqs)
        kv.rollback(named, lens)
        assert kv.lengths(ids) == [min(n for s, n in zip(named, lens) if s == i) for i in ids]
        for s in ids:
            kv.fill(s, 0, 0, rows, rows)
    kv.close()
    c.close()


def test_a_timed_step_files_every_launch_of_its_own():
    """One record per kernel of a per-stage step: set-up, embedding, six a layer, final norm, LM head, acceptance."""
    c = harness.Case(synth.TINY, torch.bfloat16, [40, 17], 3, seed=5, cache="fill").gpu_setup()
    for name, value in (("step_impl", 0), ("graph", 0), ("timing", 1)):
        c.target.set_option(name, value)
    c.run_gpu(0, debug=False)
    assert c.target.kernel_time("plan")[1] == c.target.kernel_time("embed_norm")[1] == 1
    assert c.target.kernel_time("")[1] == 2 + 6 * synth.TINY.n_layers + 3
    c.close()
