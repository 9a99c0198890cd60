"""The spans a caller passes reach C as sq_span[] whatever form they have."""
import ctypes

import numpy as np
import pytest

import paper_2602_22603_gb300 as sq


@pytest.mark.parametrize("spans", [
    [(0, 5)],
    ((1, 2), [3, 7], (2 ** 31 - 1, -(2 ** 31))),
    np.array([[4, 9], [12, 40]], dtype=np.int64),
    [(np.int32(3), np.int64(8)), (1.0, 2.9)],
    [(2 ** 31, -(2 ** 31) - 1), (2 ** 40 + 6, -(2 ** 33))],  # wrapped, as a C int
])
def test_span_forms(spans):
    want = (sq.sq_span * len(spans))(*[sq.sq_span(int(a), int(b)) for a, b in spans])
    at, keep = sq._spans(spans)
    assert keep is not None
    assert ctypes.string_at(at, ctypes.sizeof(want)) == bytes(want)


def test_no_spans():
    assert sq._spans(()) == (None, None)
    assert sq._spans([]) == (None, None)


@pytest.mark.parametrize("spans, error", [([(1,)], ValueError), ([(1, 2, 3)], ValueError),
                                          ([("a", 2)], ValueError), ([(None, 2)], TypeError),
                                          (3, TypeError)])
def test_refused_spans(spans, error):
    with pytest.raises(error):
        sq._spans(spans)
