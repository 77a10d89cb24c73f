"""The cap on the turns that empty a warp's union queue in shared memory: one
climb of the split-one rule, step by step as csrc/smem_cc.cuh takes it, ends
below the bound that the cap is built from, on the deepest trees the ids allow;
every drain loop of the kernel carries the cap."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_11839_gb300", "csrc",
                   "smem_cc.cuh")


def _climb(P, u, v):
    turns = 0
    while True:
        turns += 1
        a, b = P[u], P[v]
        hi, lo = max(a, b), min(a, b)
        ru = v if a < b else u
        if hi == lo:
            return turns
        if ru == hi:
            P[ru] = lo
            return turns
        P[ru] = P[hi]
        u, v = hi, (u if a < b else v)


@pytest.mark.parametrize("step", [1, 2, 3])
def test_deepest_climbs_stay_below_the_bound(step):
    n = 1 << 16
    P = [max(0, i - step) for i in range(n)]          # `step` chains over all ids, met at their far ends
    if step > 1:
        for k in range(step):
            P[k] = k
    assert _climb(P, n - 1, n - 2) < 1 << 18
    assert P[n - 1] <= n - 1 - step


def test_every_drain_loop_is_capped():
    text = open(SRC).read()
    assert int(re.search(r"SMEM_TURNS = 1u << (\d+);", text).group(1)) >= 21
    assert not re.search(r"while\s*\(\s*cnt", text)
    assert len(re.findall(r"\bdrain\(min\(", text)) == 1 and "left = SMEM_TURNS; cnt >= low; --left" in text
