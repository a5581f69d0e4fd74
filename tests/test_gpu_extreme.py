"""The extreme field selected on the device against the host's own selection
from the records and their maxima: the first m fields of a point by index and
then by ring position (two runs over one range with different seeds give
records that share their indices), the first of the largest maxima, too few
fields, and a limit on the records looked at.  The same kernel makes both
maxima, so everything is equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_16952_gb300 import _build
    _build.build()
    import paper_2411_16952_gb300 as T
    return T


@pytest.mark.parametrize("K,n", [(3, 700), (8, 1 << 17), (32, 1 << 15), (100, 1 << 13)])
def test_device_selection_equals_host_selection(T, K, n):
    pts = [T.make_point(1.0, 1.0, 3.0, T.PROPOSAL_PAPER, point_id=p) for p in range(3)]
    S = T.Sampler(K, pts, sample_capacity=6 * n)
    start = [(1 << 33) - 300, 0, 5]
    for seed in (1, 2):
        S.run_ranges(start, [n, n // 7 + 1, 0], seed)
    for limit in (6 * n, n):
        rec = S.samples(limit)
        umax, jm = S.field_maxima(limit)
        for point in range(4):
            sel = np.nonzero(rec["point"] == point)[0]
            sel = sel[np.argsort(rec["idx"][sel], kind="stable")]
            for m in sorted({1, 2, 33, len(sel) // 2, len(sel) - 1, len(sel), len(sel) + 1} - {0, -1}):
                ev = S.extreme_field(m, point, limit)
                if m > len(sel):
                    assert ev is None
                    continue
                b = sel[:m][int(np.argmax(umax[sel[:m]]))]
                assert ev["idx"] == rec["idx"][b] and ev["umax"] == umax[b]
                assert ev["xi"] == -np.pi + np.pi * jm[b] / K
                assert np.array_equal(ev["xhat"], rec["xhat"][b].astype(np.float64))
    S.close()
