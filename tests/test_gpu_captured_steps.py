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
    c = harness.Case(synth.TINY, torch.bfloat16, [30, 17], 4, seed=26, cache="fill").gpu_setup()
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
