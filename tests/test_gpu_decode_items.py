"""Decode where a CTA closes many items and merges runs while it streams the
next ones: short sequences dealt to few CTAs, items of one stage, two passes of
rows (G = 16, groups of forks), runs of many lengths; against the oracle and
bit for bit from call to call."""
import pytest
import torch

import paper_2602_22603_gb300 as sq
from tests.gpu_harness import Pair, assert_budget, bf16_normal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2602_22603_gb300 import build
    build.build_libsq()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (Hq, Hkv, d, page, CTAs, context lengths, forks of each)
@pytest.mark.parametrize("Hq,Hkv,D,P,ctas,lengths,forks", [
    (32, 8, 128, 64, 5, [1, 63, 64, 65, 129, 700, 3, 200], 0),   # ~13 units per CTA
    (32, 8, 128, 64, 152, [250, 900, 1800, 4000], 1),            # main + fork: 8 rows
    (32, 2, 128, 64, 40, [3000, 70], 0),                         # G = 16: two passes of rows
    (16, 4, 64, 16, 60, [1000, 1001], 3),                        # four holders: two passes, small pages
    (8, 8, 64, 8, 33, [400, 77, 8], 1),                          # G = 1, 8-token pages
    (6, 2, 128, 256, 200, [9000], 2),                            # G = 3: runs of ~60 entries
    (16, 1, 128, 64, 152, [20000], 0),                           # one KV head: 152 entries, G = 16
])
def test_items_and_runs(Hq, Hkv, D, P, ctas, lengths, forks):
    pages = sum(n // P + 4 + 2 * forks for n in lengths) + 16
    p = Pair(1, Hq, Hkv, D, P, num_pages=pages, decode_ctas=ctas, seed=Hq + P + ctas)
    keep, seqs = [], []
    try:
        for n in lengths:
            m = p.seq_new()
            keep.append(p.append(m, n))
            seqs.append(m)
            for k in range(forks):
                f = p.fork(m)
                keep.append(p.append(f, 1 + 5 * k))
                seqs.append(f)
        q_cpu = bf16_normal((len(seqs), Hq, D), ctas)
        q = q_cpu.cuda()
        exp, budget = p.oracle_decode_budget(seqs, 0, 0.1, q_cpu)
        # the first call plans, the others start early on the kept plan
        outs = [p.decode(seqs, 0, 0.1, q) for _ in range(4)]
        torch.cuda.synchronize()
        assert p.cache.sync_status() == sq.SQ_OK
        assert_budget(outs[0], exp, budget)
        assert all(torch.equal(outs[0], o) for o in outs[1:])
    finally:
        p.close()
