"""The arrival word of a decode run (CPU): whatever the order of claims and
releases, and also when the merger gives up its wait before every release has
come, the word is zero once the call is done, so the next call with the same
plan starts from zero."""
import ctypes
import random

import pytest

from tests.hostlib import lib

RELEASE = 0x10000


@pytest.mark.parametrize("n", [1, 2, 3, 19, 152, 40000, 65535])
@pytest.mark.parametrize("seed", range(3))
def test_word_ends_a_call_at_zero(n, seed):
    L = lib()
    L.sqh_arrive_leave.restype = ctypes.c_uint32
    L.sqh_arrive_leave.argtypes = L.sqh_arrive_complete.argtypes = [ctypes.c_uint32] * 2
    rng = random.Random(seed)
    word = late = 0
    for claim in range(1, n):
        word += 1
        if rng.random() < (0.0, 0.9, 1.0)[seed]:   # the claimant's release comes in time
            word += RELEASE
            assert not L.sqh_arrive_complete(word, n) or claim == n - 1
        else:
            late += 1
    assert word & 0xffff == n - 1                  # the next claim is the merger's
    word += 1
    assert bool(L.sqh_arrive_complete(word, n)) == (late == 0)
    before = rng.randint(0, late)                  # releases that come while it waits
    word += before * RELEASE
    word = L.sqh_arrive_leave(word, n)
    for _ in range(late - before):
        word = (word + RELEASE) & 0xffffffff
    assert word == 0
