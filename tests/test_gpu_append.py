"""Appends against the oracle, bit for bit, where the append kernels can go
wrong: the edges of a block's chunk of tokens, head counts that do not divide a
block's rows, page edges, more pages than one launch takes, copy-on-write of the
last page in the same launch, and batches whose holders of a page differ in fill."""
import pytest
import torch

import paper_2602_22603_gb300 as sq
from tests.gpu_harness import Pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2602_22603_gb300 import build
    build.build_libsq()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# (KV heads, d, page, tokens a block takes): 2048 / (KV heads x d / 8), at least 1
@pytest.mark.parametrize("Hkv,D,P,chunk", [
    (8, 128, 64, 16), (3, 128, 16, 42), (5, 64, 256, 51), (1, 64, 8, 256), (40, 128, 32, 3),
    (150, 128, 64, 1),
])
def test_append_sizes_and_copy_on_write(Hkv, D, P, chunk):
    p = Pair(2, Hkv, Hkv, D, P, num_pages=12 * chunk // P + 60, seed=Hkv + P)
    keep = []
    a = p.seq_new()
    for n in (1, chunk - 1, chunk, chunk + 1, P - 1, P, 2 * chunk + P + 3):
        if n > 0:
            keep.append(p.append(a, n))
    if p.cache.seq_info(a)[0] % P == 0:
        keep.append(p.append(a, 1))
    # a shared partial page: the first append copies it, the second writes in place
    b = p.fork(a)
    keep.append(p.append(b, chunk + 1))
    keep.append(p.append(a, 1))
    # and in one batch: two of the three holders copy it in the batch's launch
    c, d = p.fork(a), p.fork(a)
    keep.append(p.append_batch([c, b, a, d]))
    keep.append(p.append_batch([a, d, c]))
    assert p.cache.sync_status() == sq.SQ_OK
    p.check_tables()
    for h in (a, b, c, d):
        p.check_contents(h)
    p.close()


# Three holders of one last page with 5, 3 and 1 rows of it: whoever is left alone
# with the page writes in place, in a longer holder's rows if it is a shorter one.
# Enough planes (768 blocks a copy) that a launch's blocks overlap.
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0), (1, 0, 2), (0, 2), (2, 0)])
def test_batch_of_holders_with_different_fills(order, ragged):
    p = Pair(48, 8, 8, 128, 64, num_pages=60, seed=len(order) + 2 * ragged)
    keep = []
    for _ in range(3):
        a = p.seq_new()
        keep.append(p.append(a, 69))
        hs = [a, p.fork(a), p.fork(a)]
        p.evict(hs[1], [(67, 69)], ragged=ragged)
        p.evict(hs[2], [(65, 69)], ragged=ragged)
        if len(order) == 2:
            p.release(hs.pop(1))
            hs.insert(1, None)
        keep.append(p.append_batch([hs[i] for i in order]))
        keep.append(p.append_batch([hs[i] for i in order]))
    assert p.cache.sync_status() == sq.SQ_OK
    p.check_tables()
    for h in p.o:
        p.check_contents(h)
    p.close()


@pytest.mark.parametrize("pages", [511, 512, 513, 1030])
def test_append_more_pages_than_a_launch_takes(pages):
    P = 8
    p = Pair(1, 2, 1, 64, P, num_pages=pages + 8, seed=pages)
    a = p.seq_new()
    keep = [p.append(a, 5)]
    b = p.fork(a)
    keep.append(p.append(b, (pages - 1) * P + 2))   # copies the shared page first
    assert p.cache.sync_status() == sq.SQ_OK
    p.check_tables()
    p.check_contents(a)
    p.check_contents(b)
    p.close()
