"""Paired projections whose K is shared by the two to four pairs of a cluster, against the oracle: uneven K shares, an odd
last tile whose partner has no features, row blocks wider than the rows, several row blocks with a partial last one, more
items than clusters.  And captured steps of two caches of one target."""
import numpy as np
import pytest
import torch

import harness
from oracle import sj_oracle as orc
from paper_2510_02329_b200 import synth

pytestmark = pytest.mark.gpu

LONG_K = synth.ModelShape("long-k", 2, 2048, 16, 2, 128, 8192, 2048)                      # 8 row-parallel tiles, K 2048 and 8192
ODD = synth.ModelShape("odd-tiles", 2, 1152, 8, 2, 128, 4160, 1920, qkv_bias=True)        # 9, 12, 65 and 15 tiles; K blocks 18, 16, 65


@pytest.mark.parametrize("shape,n,gamma", [(LONG_K, 1, 1), (LONG_K, 2, 8), (LONG_K, 15, 8), (LONG_K, 29, 8), (ODD, 1, 4), (ODD, 4, 8), (ODD, 13, 12)],
                         ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_split_projections(shape, n, gamma):
    lens = [3 + 61 * b for b in range(n)]
    case = harness.Case(shape, torch.bfloat16, lens, gamma, seed=14, cache="fill").gpu_setup(max_rows=n * (gamma + 1))
    try:
        case.target.set_option("step_impl", 0)
        for mode in (orc.GREEDY, orc.SAMPLING):
            v, f = case.run_oracle(mode)
            rep = harness.compare(case, v, f, case.run_gpu(mode), mode)
            assert rep.exact + rep.margin == n
            assert rep.max_hidden_err < 2e-3, rep   # what the two activation planes leave elsewhere in these tests
    finally:
        case.close()


def test_exchanges_that_one_split_receives_in():
    """Down has 67 tiles and 286 K blocks: with 48 rows its clusters of three pairs take two items each (B200), and the second
    epilogue group's only chunk belongs to the first split, so the others finish an exchange without waiting."""
    shape = synth.ModelShape("wide-down", 1, 67 * 128, 2, 1, 128, 143 * 128, 512)
    case = harness.Case(shape, torch.bfloat16, [3 + 61 * b for b in range(8)], 5, seed=19, cache="fill", gen_device="cuda").gpu_setup(max_rows=48)
    try:
        v, f = case.run_oracle(orc.GREEDY)
        want = np.stack([x.hidden for x in f])
        off = lambda g: np.linalg.norm(g["hidden"] - want)
        case.target.set_option("step_impl", 1)
        persistent = case.run_gpu(orc.GREEDY)      # no exchange; off by as much, up to 3.2e-3: the fp16 copies of the block's own rows
        case.target.set_option("step_impl", 0)
        runs = [case.run_gpu(orc.GREEDY) for _ in range(20)]
        rep = harness.compare(case, v, f, runs[0], orc.GREEDY)
        assert rep.exact + rep.margin == 8
        assert off(runs[0]) <= 1.1 * off(persistent)
        for again in runs[1:]:
            np.testing.assert_array_equal(again["hidden"], runs[0]["hidden"])
    finally:
        case.close()


def test_captured_steps_belong_to_their_cache():
    """Two caches of one target, the same call on both in turn: a captured step holds its cache's pointers."""
    from paper_2510_02329_b200 import binding
    case = harness.Case(LONG_K, torch.bfloat16, [200, 90], 4, seed=15, cache="fill").gpu_setup()
    first = case.kv
    other = binding.KVCache(case.target, 2, 40)
    try:
        for b in range(2):
            for layer, (k, v) in enumerate(case.cache_t[1 - b]):
                other.fill(b, layer, 0, k.cuda().contiguous(), v.cuda().contiguous())
        other.set_len([0, 1], [90, 200])

        def hidden(kv):
            case.kv = kv
            return case.run_gpu(orc.GREEDY)["hidden"]

        case.target.set_option("step_impl", 0)
        case.target.set_option("graph", 0)
        want = [hidden(kv) for kv in (first, other)]
        case.target.set_option("graph", 1)
        for _ in range(2):
            for kv, w in zip((first, other), want):
                np.testing.assert_array_equal(hidden(kv), w)
    finally:
        case.kv = first
        other.close()
        case.close()
