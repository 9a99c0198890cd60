"""What one launch of sq_append_kv_batch may hold (CPU): holders of one last page
with different fills, so that one sequence writes in place to rows that another
copies.  The blocks of a launch run in any order, so the contents have to be the
oracle's with a launch's copies first and with them last."""
import ctypes
import random

import numpy as np
import pytest

import paper_2602_22603_gb300 as sq
from oracle import cache_model as ocm
from tests import fakelib

L, HKV, D = 2, 2, 64


class Caches:
    """A library cache over the stand-in and an oracle cache, in step; a token's
    rows hold its id."""

    def __init__(self, P, num_pages, copies_last):
        fakelib.lib().fake_reset()
        fakelib.lib().fake_copies_last(int(copies_last))
        self.P, self.num_pages = P, num_pages
        self.cache = sq.Cache(L, HKV, HKV, D, P, num_pages, max_seqs=200)
        self.oracle = ocm.OracleCache(num_pages, P)
        self.o = {}

    def new(self, n):
        h = self.cache.seq_new()
        self.o[h] = self.oracle.seq_new()
        k, v = self._rows(self.oracle.append(self.o[h], n))
        self.cache.append_kv(h, n, k.ctypes.data, v.ctypes.data, 1)
        return h

    def fork(self, h):
        f = self.cache.fork_aux(h)
        self.o[f] = self.oracle.fork(self.o[h])
        return f

    def evict(self, h, spans, ragged):
        self.oracle.evict(self.o[h], spans, mode="ragged" if ragged else "dense")
        (self.cache.evict_spans_ragged if ragged else self.cache.evict_spans)(h, spans, 1)

    def append_batch(self, hs):
        k, v = self._rows([self.oracle.append(self.o[h], 1)[0] for h in hs])
        self.cache.append_kv_batch(hs, k.ctypes.data, v.ctypes.data, 1)

    def _rows(self, ids):
        k = np.empty((L, len(ids), HKV, D), np.uint16)
        k[:] = np.asarray(ids, np.uint16)[None, :, None, None]
        k += (np.arange(L, dtype=np.uint16) * 1000)[:, None, None, None]
        return k, k + np.uint16(30000)

    def check(self):
        shape = (L, self.num_pages, 2, HKV, self.P, D)
        mem = (ctypes.c_uint16 * int(np.prod(shape))).from_address(sq.sq_pool_ptr(self.cache.handle))
        pool = np.frombuffer(mem, np.uint16).reshape(shape)
        for h, o in self.o.items():
            assert self.cache.page_table(h) == self.oracle.page_table(o)
            fills = self.cache.page_fills(h)
            assert fills == self.oracle.page_fills(o)
            page = np.repeat(self.cache.page_table(h), fills)
            slot = np.concatenate([np.arange(f) for f in fills])
            k, v = self._rows(self.oracle.tokens(o))
            assert np.array_equal(pool[:, page, 0, :, slot].transpose(1, 0, 2, 3), k), h
            assert np.array_equal(pool[:, page, 1, :, slot].transpose(1, 0, 2, 3), v), h


@pytest.fixture
def caches(monkeypatch):
    monkeypatch.setattr(sq, "_lib", fakelib.lib())
    made = []

    def make(*args):
        made.append(Caches(*args))
        return made[-1]

    yield make
    for c in made:   # while the stand-in is the library
        c.cache.close()


@pytest.mark.parametrize("copies_last", [False, True])
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0), (1, 0, 2), (0, 2), (2, 0)])
def test_holders_of_different_fills(caches, order, ragged, copies_last):
    c = caches(64, 40, copies_last)
    a = c.new(69)                       # last page: 5 rows
    hs = [a, c.fork(a), c.fork(a)]
    c.evict(hs[1], [(67, 69)], ragged)  # 3 rows, the page still shared
    c.evict(hs[2], [(65, 69)], ragged)  # 1 row
    if len(order) == 2:
        c.cache.release(hs[1], 1)
        c.oracle.release(c.o.pop(hs[1]))
    c.append_batch([hs[i] for i in order])
    c.check()
    c.append_batch([hs[i] for i in order])
    c.check()
    # the common step stays one launch
    assert fakelib.lib().fake_count(fakelib.APPEND_BATCH) <= 3


@pytest.mark.parametrize("copies_last", [False, True])
@pytest.mark.parametrize("seed", range(6))
def test_random_holders(caches, seed, copies_last):
    rng = random.Random(seed)
    c = caches(rng.choice([8, 64]), 900, copies_last)
    live = []
    for _ in range(rng.choice([3, 40])):
        live.append(c.new(rng.randint(1, 100)))
    while len(live) < 150:
        live.append(c.fork(rng.choice(live)))
    for _ in range(4):
        for h in rng.sample(live, 60):
            n = c.cache.seq_info(h)[0]
            tail = c.cache.page_fills(h)[-1]
            if tail > 1:
                c.evict(h, [(n - rng.randint(1, tail - 1), n)], rng.random() < 0.5)
        c.append_batch(rng.sample(live, rng.choice([2, 64, 65, 150])))
        c.check()


def test_equal_fills_take_one_launch(caches):
    c = caches(64, 60, True)
    a = c.new(70)
    hs = [a] + [c.fork(a) for _ in range(9)]
    c.append_batch(hs)
    assert fakelib.lib().fake_count(fakelib.APPEND_BATCH) == 1
    c.check()
