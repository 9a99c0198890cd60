"""What an attention call that fails after its upload leaves behind (CPU): the
calls that follow, on whatever stream, use its plan and its workspace only after
what it had enqueued."""
import pytest

import paper_2602_22603_gb300 as sq
from tests import fakelib

HQ, HKV, D, P = 8, 2, 128, 64
Q, OUT = 1 << 20, 2 << 20  # never read or written by the stand-in


@pytest.fixture
def cache(monkeypatch):
    monkeypatch.setattr(sq, "_lib", fakelib.lib())
    fakelib.lib().fake_reset()
    c = sq.Cache(1, HQ, HKV, D, P, 200)
    yield c
    c.close()


def seq(c, n):
    h = c.seq_new()
    import numpy as np
    k = np.zeros((1, n, HKV, D), np.uint16)
    c.append_kv(h, n, k.ctypes.data, k.ctypes.data, 1)
    return h


def prefill(c, h, stream, n_q=8):
    c.prefill_attention(h, 0, n_q, Q, OUT, sq.SQ_OUT_BF16, None, 0.1, (), stream)


def decode(c, h, stream):
    c.decode_attention([h], 0, Q, OUT, sq.SQ_OUT_BF16, 0.1, stream)


@pytest.mark.parametrize("call", [prefill, decode])
def test_streams_take_turns(cache, call):
    a, b = seq(cache, 3000), seq(cache, 2000)
    for _ in range(2):
        for stream in (1, 2, 3):
            for h in (a, b):
                call(cache, h, stream)
    assert fakelib.lib().fake_races() == 0


def test_prefill_without_room_for_partial_results(cache):
    L = fakelib.lib()
    a, b, c = seq(cache, 3000), seq(cache, 500), seq(cache, 9000)
    prefill(cache, b, 1)                   # split in few pieces: a small workspace
    assert L.fake_count(fakelib.COMBINE) == 1
    L.fake_malloc_limit(1 << 20)
    prefill(cache, a, 1)                   # no room for its pieces: not split
    prefill(cache, a, 2)
    prefill(cache, c, 2)
    assert L.fake_count(fakelib.COMBINE) == 1
    prefill(cache, b, 2)                   # ... nor the first call's any more
    assert L.fake_count(fakelib.COMBINE) == 1 and L.fake_count(fakelib.PREFILL) == 5
    L.fake_malloc_limit(-1)
    prefill(cache, c, 3, n_q=9)            # room again
    prefill(cache, b, 1)
    assert L.fake_count(fakelib.COMBINE) == 2
    assert L.fake_races() == 0


@pytest.mark.parametrize("kind,call", [
    (fakelib.PREFILL, prefill), (fakelib.COMBINE, prefill), (fakelib.DECODE, decode)])
@pytest.mark.parametrize("same", [True, False])
def test_after_a_failed_launch(cache, kind, call, same):
    L = fakelib.lib()
    a, b = seq(cache, 3000), seq(cache, 2000)
    L.fake_fail(kind)
    with pytest.raises(sq.SqError) as e:
        call(cache, a, 1)
    assert e.value.code == sq.SQ_ERR_CUDA and L.fake_count(kind) == 1
    call(cache, a if same else b, 2)   # the call again, or another one
    call(cache, a, 3)
    assert L.fake_count(kind) == 3
    assert L.fake_races() == 0
    # and where the plan was in use before
    L.fake_fail(kind)
    with pytest.raises(sq.SqError):
        call(cache, a, 1)
    call(cache, b, 2)
    call(cache, a, 2)
    call(cache, a, 1)
    assert L.fake_races() == 0
