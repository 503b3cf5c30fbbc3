"""The exchange between the splits of a paired projection, as a state machine: whatever the order in which the splits of a
cluster get to run, no wait misses its phase and none is passed early.  The number of "my sums have been read" barriers is read
from the kernel's source."""
import itertools
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_02329_b200", "csrc", "sj_gemm_pair.cuh")
ARM, WAIT_FREE, SEND, WAIT_FULL, ARRIVE = range(5)


def free_bars_of_the_kernel():
    m = re.search(r"constexpr int kPairFreeBars = (\d+);", open(SRC).read())
    return int(m.group(1)) if m else 1


def failure(S, receivers, F):
    """A reachable state of S splits and one exchange per entry of `receivers` (the splits that finish chunks of it) in which a
    wait is passed before its phase is complete or nobody can go on; None if there is none.  An mbarrier wait knows the parity only."""
    N = len(receivers)
    # a split's program counter is 5 n + the step of exchange n that it does next; everything else follows from the counters
    steps = lambda pc, op: max(0, (pc - op + 4) // 5)                       # how often it has done `op`
    def free_arrivals(pcs, f, bar):
        return sum(len(range(bar, steps(pc, ARRIVE), F)) for j, pc in enumerate(pcs) if j != f)

    def full_phases(pcs, f):
        n = 0
        while n < steps(pcs[f], ARM) and (f not in receivers[n] or all(steps(pc, SEND) > n for j, pc in enumerate(pcs) if j != f)):
            n += 1
        return n

    def can_go(pcs, f):
        n, op = divmod(pcs[f], 5)
        if op == WAIT_FREE and n > 0:
            k, phases = (n - 1) // F, free_arrivals(pcs, f, (n - 1) % F) // (S - 1)
        elif op == WAIT_FULL:
            k, phases = n, full_phases(pcs, f)
        else:
            return True
        if phases % 2 == k % 2:                                             # the running phase has the parity that is waited for
            return False
        assert phases > k, ("passed early", pcs, f)
        return True

    seen, todo = {(0,) * S}, [(0,) * S]
    while todo:
        pcs = todo.pop()
        nexts = [pcs[:f] + (pcs[f] + 1,) + pcs[f + 1:] for f in range(S) if pcs[f] < 5 * N and can_go(pcs, f)]
        if not nexts and any(pc < 5 * N for pc in pcs):
            return pcs
        for x in nexts:
            if x not in seen:
                seen.add(x)
                todo.append(x)
    return None


def chunk_sets(S):
    """Who finishes chunks of a row block of 0 .. 4 of them: chunk j belongs to split j % S."""
    return sorted({frozenset(j % S for j in range(n)) for n in range(5)}, key=len)


@pytest.mark.parametrize("S,N", [(2, 5), (3, 4), (4, 2)])
def test_no_order_of_the_splits_misses_a_phase(S, N):
    F = free_bars_of_the_kernel()
    for receivers in itertools.product(chunk_sets(S), repeat=N):
        assert failure(S, receivers, F) is None, (S, [sorted(r) for r in receivers])


def test_the_model_sees_a_phase_that_is_overtaken():
    """One barrier, two exchanges that only split 0 receives in: its partner may arrive twice before it looks."""
    assert failure(2, [frozenset({0})] * 3, 1) is not None
    assert failure(2, [frozenset({0, 1})] * 3, 1) is None                   # both receive: nobody runs ahead
