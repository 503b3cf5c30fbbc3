"""The host loop's device buffers: they follow the attributes that a cycle reads, and nobody gets their memory while a queued pass
still writes it."""
import pytest
import torch

from paper_2510_02329_b200 import loop, synth
from test_gpu_extensions import _target_and_cache

pytestmark = pytest.mark.gpu


@pytest.fixture
def pair():
    """A target, the same model as its own draft, and a third copy to decode alone; fp32, so every draft is accepted."""
    made = [_target_and_cache(synth.TINY, torch.float32, 0, 2)[1:] for _ in range(3)]
    yield made
    torch.cuda.synchronize()
    for target, kv in made:
        kv.close()
        target.close()


def test_cycles_follow_gamma_and_the_sequences(pair):
    (draft, draft_kv), (target, target_kv), (solo, solo_kv) = pair
    prompts = [[int(t) for t in synth.token_ids(synth.TINY.vocab, n, seed=60 + n, stream=3)] for n in (9, 5)]
    dec = loop.SpeculativeDecoder(draft, draft_kv, target, target_kv, [0, 1], 4)
    dec.prefill(prompts)
    got = [[], []]
    for gamma in (4, 7, 2, 5):
        dec.gamma = gamma
        for o, p in zip(got, dec.cycle(use_judge=False)):
            assert len(p) == gamma + 1
            o.extend(p)
    dec.seq_ids, dec.B, dec.lens, dec.pending = [1], 1, dec.lens[1:], dec.pending[1:]
    got[1].extend(dec.cycle(use_judge=False)[0])
    for s in (0, 1):
        assert got[s] == loop.greedy_decode(solo, solo_kv, s, prompts[s], len(got[s]))


def test_a_queued_pass_keeps_its_buffers(pair):
    """A cycle that accepts everything ends with a draft pass that nobody waits for: while it is held back, no new tensor of the
    same size gets the memory that it will write."""
    (draft, draft_kv), (target, target_kv), _ = pair
    dec = loop.SpeculativeDecoder(draft, draft_kv, target, target_kv, [0, 1], 3)
    dec.prefill([[int(t) for t in synth.token_ids(synth.TINY.vocab, n, seed=60 + n, stream=3)] for n in (9, 5)])
    dec.cycle(use_judge=False)
    plain = loop.SpeculativeDecoder._decode

    def held_back(target, kv, seqs):
        with torch.cuda.stream(target.stream):
            torch.cuda._sleep(200_000_000)            # about a tenth of a second on the draft's stream
        return plain(target, kv, seqs)

    dec._decode = held_back
    dec.cycle(use_judge=False)
    got = [torch.full((2,), -7, dtype=torch.int32, device="cuda") for _ in range(64)]
    got += [torch.full((2, 1), -7.0, device="cuda") for _ in range(64)]
    torch.cuda.synchronize()
    assert all(bool((t == -7).all()) for t in got)


def test_a_draft_pass_that_timed_out_is_reported():
    from paper_2510_02329_b200 import binding
    shape = synth.ModelShape("gqa-small", 3, 256, 4, 2, 64, 512, 1024, rope_theta=5e5)
    (_, target, target_kv), (_, draft, draft_kv) = (_target_and_cache(shape, torch.bfloat16, 0, 1) for _ in range(2))
    try:
        dec = loop.SpeculativeDecoder(draft, draft_kv, target, target_kv, [0], 3)
        dec.prefill([[int(t) for t in synth.token_ids(shape.vocab, 9, seed=60, stream=3)]])
        draft.expire_wait(0)
        with pytest.raises(binding.SjError) as e:
            dec.cycle()
        assert e.value.status == 7
    finally:
        target_kv.close(); draft_kv.close(); target.close(); draft.close()
