"""Arguments of Sampler.extreme_field that a C integer does not hold as they
are: a point or a count above its range, a point that is not an int."""
import ctypes as C

import numpy as np
import pytest

import paper_2411_16952_gb300 as T


@pytest.fixture
def sampler(monkeypatch):
    """A handle of two points with 100 and 40 fields, cut as C cuts its arguments."""
    def fake(h, K, point, m, max_records):
        point, m = C.c_int(point).value, C.c_uint64(m).value
        n = {0: 100, 1: 40}.get(point, 0)
        return n, (10 * point + m, 1.5, 0, np.zeros(2 * K, np.float32)) if n >= m else None
    monkeypatch.setattr(T, "sampler_extreme_field", fake)
    S = object.__new__(T.Sampler)
    S.h, S.K, S.n_points = None, 4, 2
    return S


@pytest.mark.parametrize("point,m,idx", [(0, 50, 50), (1, 30, 40), (1.0, 30, 40), (np.float32(1), np.int64(30), 40),
                                         (1 << 32, 30, None), ((1 << 32) + 1, 30, None), (-1, 30, None), (2, 30, None),
                                         (0.5, 30, None), (0, (1 << 64) + 1, None), (0, 1 << 64, None),
                                         (0, 101, None), (1, -10, 40)])
def test_point_and_count_as_numbers(sampler, point, m, idx):
    got = sampler.extreme_field(m=m, point=point)
    assert (got is None) if idx is None else got["idx"] == idx


def test_no_fields_are_refused(sampler):
    for m in (0, -100, -(1 << 65)):
        with pytest.raises(ValueError):
            sampler.extreme_field(m=m, point=0)
