"""Evictions whose plan goes with the launch and evictions whose plan is read
from memory, at the sizes where the one becomes the other (224 records)."""
import pytest
import torch

from tests.gpu_harness import Pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2602_22603_gb300 import build
    build.build_libsq()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# ragged: every span is a window of its own, with three tiles (32 and 12 rows
# moved, 10 zeroed) and two pieces; dense: the rows from the first span on, 32 a
# tile, a tile and one or two pieces each
@pytest.mark.parametrize("ragged,count", [(True, 1), (True, 44), (True, 45), (True, 90),
                                          (False, 1), (False, 13), (False, 14), (False, 40)])
@pytest.mark.parametrize("forked", [False, True])
def test_plan_sizes(ragged, count, forked):
    P, n = 64, 4 * 64 * count + 30
    p = Pair(2, 8, 2, 128, P, num_pages=3 * (n // P + 2) + 8, seed=count, physical=ragged)
    try:
        h = p.seq_new()
        keep = [p.append(h, n)]
        if forked:
            f = p.fork(h)
            keep.append(p.append(f, 5))
        p.evict(h, [(4 * P * i + 10, 4 * P * i + 20) for i in range(count)], ragged=ragged)
        p.check_tables()
        p.check_contents(h)
        if forked:
            p.check_contents(f)
        if ragged:
            p.check_zero_slots()
        torch.cuda.synchronize()
        assert p.cache.sync_status() == 0
    finally:
        p.close()
