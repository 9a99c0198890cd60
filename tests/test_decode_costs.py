"""Decode plans and the units' start-up costs (CPU): the items tile every
(segment, KV head) once and in order, and the CTAs' shares of the cost line are
even."""
import random

import pytest

from tests.hostlib import HostCache

UNIT, SHORT, SHORT_STAGES = 4, 8, 2


@pytest.mark.parametrize("seed", range(8))
def test_items_tile_the_cost_line(seed):
    rng = random.Random(seed)
    Hkv = rng.choice([1, 2, 8])
    hc = HostCache(1, 4 * Hkv, Hkv, 128, 64, 4000, max_seqs=64)
    seqs = []
    for _ in range(rng.randint(1, 6)):
        rc, h = hc.seq_new()
        assert hc.append(h, rng.choice([1, 60, 64, 65, 130, rng.randint(1, 9000)])) == 0
        seqs.append(h)
        if rng.random() < 0.6:
            rc, a = hc.fork(h)
            assert hc.append(a, rng.randint(1, 64)) == 0
            seqs.append(a)
    n_ctas = rng.choice([1, 7, 152])
    rc, plan = hc.plan_decode(seqs, n_ctas)
    assert rc == 0
    stages = [-(-s["n_tok"] // 64) for s in plan["segs"]]
    at = {}
    cb = plan["cta_begin"]
    share = []
    for c in range(len(cb) - 1):
        cost = 0
        for i in range(cb[c], cb[c + 1]):
            seg, head, s0, s1 = plan["items"][i]
            assert s0 == at.get((seg, head), 0) and s1 > s0
            at[seg, head] = s1
            cost += s1 - s0
            if s0 == 0:
                cost += SHORT if stages[seg] <= SHORT_STAGES else UNIT
        share.append(cost)
    assert all(at[s, h] == stages[s] for s in range(len(stages)) for h in range(Hkv))
    # an even cut of the line; a start-up cost may fall to either side of a cut
    assert max(share) - min(share) <= 2 * SHORT + 1
