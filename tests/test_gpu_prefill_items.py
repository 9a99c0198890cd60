"""Masked prefill where a CTA works through several items: more query units
than SMs (short and long items, empty ones, one- and two-tile and dual-key
items in one list), and a last round split in key ranges with its merge."""
import math

import numpy as np
import pytest
import torch

import paper_2602_22603_gb300 as sq
from synthetic import random_spans
from tests.gpu_harness import Pair
from tests.test_gpu_prefill import check, check_budget_rows, run_prefill

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2602_22603_gb300 import build
    build.build_libsq()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("Hq,Hkv,D,P,n,n_q,spans", [
    (100, 100, 64, 64, 300, 300, []),               # items of 2 and 3 key tiles, the last dual-key
    (100, 100, 64, 64, 300, 300, [(0, 260)]),       # the first unit of every head sees no key
    (100, 100, 128, 16, 130, 130, [(3, 40)]),       # one item per head, two tiles and 2 rows
    (200, 200, 64, 64, 100, 100, []),               # one key tile: tile b idle
    (160, 40, 128, 64, 321, 321, [(60, 190)]),      # G = 4: 6 units per head, ragged end
    (126, 42, 64, 128, 400, 190, [(0, 100)]),       # G = 3: rows that are no query
])
def test_more_units_than_sms(Hq, Hkv, D, P, n, n_q, spans):
    p = Pair(1, Hq, Hkv, D, P, num_pages=n // P + 4, seed=Hq + n)
    try:
        h = p.seq_new()
        p.append(h, n)
        check(p, h, 0, n_q, spans, seed=n + n_q)
        check(p, h, 0, n_q, spans, seed=n, out_dtype=sq.SQ_OUT_BF16)
    finally:
        p.close()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("Hkv,G", [(152, 1), (76, 2), (21, 2), (19, 4), (16, 2), (2, 8)])
def test_merges_of_few_and_many_splits(D, Hkv, G):
    # 1, 2, 7, 8, 9 and 23 or more splits of every unit (8 and less merge a row a warp)
    p = Pair(1, Hkv * G, Hkv, D, 64, num_pages=60, seed=D + Hkv)
    try:
        h = p.seq_new()
        p.append(h, 3003)
        check(p, h, 0, 5, [(100, 900)], seed=Hkv)
        check(p, h, 0, 3, [], seed=Hkv, out_dtype=sq.SQ_OUT_BF16)
    finally:
        p.close()


@pytest.mark.parametrize("D,n,n_q", [(64, 18000, 5120), (128, 18001, 5003)])
def test_split_last_round(D, n, n_q):
    # 160 units on 152 SMs: the units of a second round are split in key ranges
    p = Pair(1, 8, 8, D, 64, num_pages=n // 64 + 4, seed=D)
    try:
        h = p.seq_new()
        p.append(h, n)
        spans = random_spans(3, 5, 2500, 64, n, median=400)
        scale = 1.0 / math.sqrt(D)
        q, out, lse = run_prefill(p, h, 0, n_q, spans, n, scale)
        assert torch.isfinite(out).all() and torch.isfinite(lse).all()
        rows = sorted(set(np.linspace(0, n_q - 1, 60).round().astype(int).tolist()))
        check_budget_rows(p, h, 0, q, out, spans, scale, rows)
    finally:
        p.close()


def test_split_partials_across_streams():
    # six split plans in four plan entries, on three streams in turn: the
    # partials and the entries that every call shares pass from stream to stream
    p = Pair(1, 8, 2, 64, 64, num_pages=6 * 70 + 4, seed=11)
    try:
        hs = [p.seq_new() for _ in range(6)]
        for i, h in enumerate(hs):
            p.append(h, 4000 + 37 * i)
        g = torch.Generator(device="cuda").manual_seed(5)
        q = torch.randn(6, 16, 8, 64, device="cuda", generator=g).to(torch.bfloat16)
        n_q = [16, 9, 16, 3, 12, 16]

        def one(i, out, stream):
            p.cache.prefill_attention(hs[i], 0, n_q[i], q[i], out, sq.SQ_OUT_F32, None, 0.125,
                                      (), stream)
        want = torch.zeros(6, 16, 8, 64, device="cuda")
        for i in range(6):
            one(i, want[i], None)
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(3)]
        order = [(7 * k + k // 5) % 6 for k in range(60)]
        got = torch.zeros(len(order), 16, 8, 64, device="cuda")
        torch.cuda.synchronize()
        for k, i in enumerate(order):
            one(i, got[k], streams[k % 3].cuda_stream)
        torch.cuda.synchronize()
        for k, i in enumerate(order):
            assert torch.equal(got[k], want[i]), (k, i)
    finally:
        p.close()


@pytest.mark.parametrize("D,P,n,new,n_q,grow", [
    (128, 64, 9000, 3000, 8, True),     # one tile of queries, keys split over the SMs
    (128, 64, 9000, 40, 8, False),
    (64, 128, 5000, 1000, 12, True),
    (128, 256, 300, 200, 150, True),    # few key tiles: the ring holds an item's all
    (64, 64, 100, 1, 1, False),         # one key tile
    (128, 64, 6000, 2500, 2500, True),  # two-tile items, several per SM
    (64, 32, 3000, 600, 9, True),       # small pages: nothing is loaded early
])
def test_layers_right_after_appends(D, P, n, new, n_q, grow):
    """The calls after the first reuse its plan and load keys before the work
    before them is done: never from pages whose rows are still being written."""
    L = 3
    p = Pair(L, 8, 2, D, P, num_pages=6 * ((n + 8 * new) // P + 4), seed=n + new)
    try:
        g = torch.Generator(device="cuda").manual_seed(n)

        def rand(*shape):
            return torch.randn(*shape, device="cuda", generator=g).to(torch.bfloat16)
        kv = [(rand(L, m, 2, D), rand(L, m, 2, D)) for m in [n] + [new] * 8]
        q = rand(8, L, n_q, 8, D)
        filler = rand(L, 20000, 2, D)   # (keeps the stream busy while the calls are issued)
        spare = sq.Cache(L, 8, 2, D, 64, 340)

        def steps(sync):
            h = p.cache.seq_new()
            p.cache.append_kv(h, n, *kv[0])
            outs = []
            for i in range(8):
                if not sync:
                    x = spare.seq_new()
                    spare.append_kv(x, 20000, filler, filler)
                    spare.release(x)
                target = h if grow else p.cache.fork_aux(h)
                p.cache.append_kv(target, new, *kv[1 + i])
                for layer in range(L):
                    out = torch.empty(n_q, 8, D, device="cuda")
                    if sync:
                        torch.cuda.synchronize()
                    p.cache.prefill_attention(target, layer, n_q, q[i, layer], out, sq.SQ_OUT_F32,
                                              None, 0.1, ())
                    outs.append(out)
                if not grow:
                    p.cache.release(target)
            p.cache.release(h)
            torch.cuda.synchronize()
            assert p.cache.sync_status() == sq.SQ_OK
            return outs
        want, got = steps(True), steps(False)
        for i, (x, y) in enumerate(zip(want, got)):
            assert torch.isfinite(x).all() and torch.equal(x, y), (i // L, i % L)
        spare.close()
    finally:
        p.close()


def test_prefill_replayed_from_a_cuda_graph():
    p = Pair(2, 8, 2, 128, 64, num_pages=200, seed=3)
    try:
        h, other = p.seq_new(), p.seq_new()
        p.append(h, 6000)
        q = torch.zeros(2, 16, 8, 128, dtype=torch.bfloat16, device="cuda")
        outs = torch.zeros(2, 16, 8, 128, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())

        def layers():
            for layer in range(2):
                p.cache.prefill_attention(h, layer, 16, q[layer], outs[layer], sq.SQ_OUT_F32, None,
                                          0.1, ())
        qs = [torch.randn(2, 16, 8, 128, device="cuda").to(torch.bfloat16) for _ in range(3)]
        want = []
        with torch.cuda.stream(s):
            for x in qs:
                q.copy_(x)
                layers()
                want.append(outs.clone())
            p.append(other, 100)   # a write that no call has found complete yet
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            layers()
        for x, w in zip(qs, want):
            q.copy_(x)
            outs.fill_(float("nan"))
            g.replay()
            torch.cuda.synchronize()
            assert torch.isfinite(w).all() and torch.equal(outs, w)
        assert p.cache.sync_status() == sq.SQ_OK
        del g
    finally:
        p.close()


@pytest.mark.parametrize("Hq,Hkv,n,n_q,rise", [
    (320, 160, 1000, 3, 9.0),      # 6 rows of a warp hold queries
    (320, 160, 1000, 3, 15.0),
    (480, 160, 1000, 200, 12.0),   # G = 3: two rows of every tile hold none
])
def test_dominant_key_in_a_partly_filled_warp(Hq, Hkv, n, n_q, rise):
    """A key of an item's later tiles whose weight passes the running maximum
    by 2^9 .. 2^15 sets the maximum in warps with rows that are no query, so its
    weight is exactly 1 and the log-sum-exp is off by the rounding of the other
    weights alone: n of them, 2^-rise each, every one off by an independent 2^-9
    at most, so by less than 6 sqrt(n) 2^-rise 2^-9 together.  Rounded to bf16
    the large weight itself (2^(rise + 0.40625)) would be off by 0.0022."""
    p = Pair(1, Hq, Hkv, 64, 64, num_pages=n // 64 + 4, seed=1)
    try:
        h = p.seq_new()
        scale = math.log(2.0)      # logits in powers of two
        k = torch.zeros(1, n, Hkv, 64, dtype=torch.bfloat16, device="cuda")
        k[..., 1] = 0.11 * torch.randn(n, device="cuda").to(torch.bfloat16)[None, :, None]
        k[0, 700 if n_q < 10 else 500, :, 0] = rise + 0.40625   # (not near a power of two)
        v = torch.randn(1, n, Hkv, 64, device="cuda").to(torch.bfloat16)
        p.cache.append_kv(h, n, k, v)
        q = torch.zeros(n_q, Hq, 64, dtype=torch.bfloat16, device="cuda")
        q[..., :2] = 1
        out = torch.empty(n_q, Hq, 64, device="cuda")
        lse = torch.empty(n_q, Hq, device="cuda")
        p.cache.prefill_attention(h, 0, n_q, q, out, sq.SQ_OUT_F32, lse, scale, ())
        x = (k[0, :, 0, 0].double() + k[0, :, 0, 1].double()) * scale
        want = torch.stack([torch.logsumexp(x[:n - n_q + i + 1], 0) for i in range(n_q)])
        # the queries of the warp of 32 rows that ends a tile of BP positions
        bp = 128 // (Hq // Hkv)
        at = [i for i in range(n_q) if n_q < bp or i % bp >= 96 * Hkv // Hq]
        assert at
        err = (lse.double() - want[:, None]).abs()[at].max().item()
        assert err <= 6 * math.sqrt(n) * 2.0 ** (-rise - 9) + 2e-5, err
    finally:
        p.close()
