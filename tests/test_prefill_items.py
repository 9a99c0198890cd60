"""The prefill planner's work items (CPU): every key tile of every query unit
is in exactly one item, split units have contiguous partial results that tile
their keys, and CTAs that take the items in order finish close together."""
import ctypes
import heapq
import random

import pytest

from tests.hostlib import lib, plan_prefill


def items(Hq, Hkv, n, n_q, spans, ctas=152, P=64):
    L = lib()
    cap = 1 << 16
    info = (ctypes.c_int64 * 3)()
    it = (ctypes.c_int32 * (4 * cap))()
    mg = (ctypes.c_int32 * (3 * cap))()
    arr = (ctypes.c_int32 * max(1, 2 * len(spans)))(*[x for s in spans for x in s])
    rc = L.sqh_prefill_items(Hq, Hkv, P, n, n_q, arr, len(spans), ctas, info, it, cap, mg, cap)
    assert rc == 0
    return ([tuple(it[4 * i:4 * i + 4]) for i in range(info[0])],
            [tuple(mg[3 * i:3 * i + 3]) for i in range(info[1])], info[2])


@pytest.mark.parametrize("Hq,Hkv,n,n_q,spans", [
    (32, 8, 1, 1, []),                               # one tile
    (32, 8, 300, 300, [(0, 300)]),                   # every key masked
    (16, 4, 517, 517, [(30, 200)]),
    (32, 8, 33001, 3001, [(100, 5000)]),             # 376 units: a split last round
    (32, 8, 25501, 1500, []),                        # 192 units: 1.26 rounds
    (32, 8, 131080, 8, []),                          # one unit per head
    (32, 8, 131072, 512, []),
    (32, 8, 9000, 9000, [(50, 700), (800, 4000)]),   # causal from the start
    (6, 2, 40000, 6500, []),                         # G = 3: padded query tiles
    (32, 8, 32768, 32768, [(100, 5000)]),
    (64, 8, 60000, 2500, []),
])
def test_items_cover_every_key_tile_once(Hq, Hkv, n, n_q, spans):
    rc, info, _ = plan_prefill(Hq, Hkv, n, n_q, spans)
    assert rc == 0
    got, merges, n_parts = items(Hq, Hkv, n, n_q, spans)
    units = info["n_qt"] * Hkv
    seen = {u: [] for u in range(units)}
    for u, t0, T, part in got:
        seen[u].append((t0, T, part))
    split = {u: (p0, k) for u, p0, k in merges}
    used = []
    for u, parts in seen.items():
        parts.sort()
        at = 0
        for t0, T, _ in parts:
            assert t0 == at and T >= (1 if len(parts) > 1 else 0)
            at += T
        assert at == info["qt_tiles"][u // Hkv]
        if len(parts) == 1:
            assert parts[0][2] == -1 and u not in split
        else:
            p0, k = split[u]
            assert [p for _, _, p in parts] == list(range(p0, p0 + k)) and 2 <= k <= 64
            used += range(p0, p0 + k)
    assert sorted(used) == list(range(n_parts))


PART_LIMIT = 128 << 20           # bytes of partial results a plan may have
PART_BYTES = 2 * 128 * (128 + 1) * 4


def test_partial_results_are_bounded():
    # without a limit 1,820 and 2,272 of 132 KB each (last rounds), 2,736 (few
    # units), and 12 of the 400 drawn ones above the limit
    shapes = [(32, 2, 236067, 5976), (32, 2, 197877, 10857), (32, 8, 250000, 1150)]
    rng = random.Random(1)
    for _ in range(400):
        n = int(2 ** rng.uniform(12, 18))
        shapes.append((*rng.choice([(32, 8), (64, 8), (16, 4), (32, 2), (8, 8), (32, 4)]), n,
                       int(min(n, 2 ** rng.uniform(3, 14)))))
    most = 0
    for Hq, Hkv, n, n_q in shapes:
        _, _, n_parts = items(Hq, Hkv, n, n_q, [])
        assert n_parts * PART_BYTES <= PART_LIMIT, (Hq, Hkv, n, n_q, n_parts)
        most = max(most, n_parts)
    assert most > 700   # the limit is no tighter than it says


@pytest.mark.parametrize("n,n_q,most", [
    (33001, 3001, 1.03),    # 2.47 rounds of work: three whole rounds would be 1.21
    # 1.26 rounds (two would be 1.58): a whole unit and two sevenths of another,
    # 1.286 units at most 204 tiles long, over 1.263 of 192 .. 204: 1.07
    (25501, 1500, 1.07),
    (32768, 32768, 1.02),
    (9000, 9000, 1.06),
])
def test_ctas_finish_close_together(n, n_q, most):
    got, _, _ = items(32, 8, n, n_q, [])
    busy = [0] * 152
    for _, _, T, _ in got:
        heapq.heapreplace(busy, busy[0] + T)
    assert max(busy) <= most * sum(busy) / 152
