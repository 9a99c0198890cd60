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
