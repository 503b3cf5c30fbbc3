"""How long captured steps live: a cache takes its own along, and the oldest go when there are too many."""
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _captures(work):
    """How many graphs `work` instantiates."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU, torch.profiler.ProfilerActivity.CUDA]) as p:
        work()
        torch.cuda.synchronize()
    return sum(e.count for e in p.key_averages() if e.key.startswith("cudaGraphInstantiate"))


@pytest.fixture
def case():
    c = harness.Case(synth.TINY, torch.bfloat16, [30, 17], 4, seed=26, cache="fill").gpu_setup(max_rows=32)
    c.target.set_option("step_impl", 0)
    yield c
    c.close()


def test_destroying_a_cache_keeps_the_steps_of_others(case):
    step = lambda: case.run_gpu(orc.GREEDY)
    other = binding.KVCache(case.target, 2, 40)
    assert _captures(step) == 1
    assert _captures(step) == 0
    mine, case.kv = case.kv, other
    assert _captures(step) == 1
    case.kv = mine
    other.close()
    assert _captures(step) == 0
    v, f = case.run_oracle(orc.GREEDY)
    rep = harness.compare(case, v, f, case.run_gpu(orc.GREEDY), orc.GREEDY)
    assert rep.exact + rep.margin == 2


def test_the_oldest_captured_step_goes(case):
    """513 steps of different keys (draft length, sequences, top_k, cache), one more than a target keeps.  One that is used in between
    stays, the first one does not."""
    d = {g: torch.zeros((2, g), dtype=torch.int32, device="cuda") for g in range(1, 32)}
    caches = [binding.KVCache(case.target, 2, 8) for _ in range(6)]
    def step(kv, B, g, top_k):
        out = binding.VerifyBuffers(B, g)
        binding.verify(case.target, kv, list(range(B)), d[g][:B].contiguous(), out, commit=False, top_k=top_k)

    shapes = [(kv, B, g, k) for kv in caches for k in (0, 2) for B in (1, 2) for g in range(1, 32) if B * (g + 1) <= 32][:513]
    kept = shapes[1]
    assert len(shapes) == 513
    step(caches[0], 1, 31, 0)                               # workspaces have grown to their size: growing drops captured steps
    case.target.set_option("attn_two_term_layers", 1)       # drops what has been captured
    for i, s in enumerate(shapes):
        step(*s)
        if i % 100 == 50:
            step(*kept)
    case.target.sync()
    assert _captures(lambda: step(*kept)) == 0
    assert _captures(lambda: step(*shapes[0])) == 1
    case.target.sync()
    for kv in caches:
        kv.close()
