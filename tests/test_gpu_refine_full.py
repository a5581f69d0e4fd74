"""The FP64 pass with a full queue: from a number of queued proposals on, one
thread takes a proposal where the lanes of a batch would not all have a mode,
and SIR runs whose ring is smaller than the queue take that form too.  One run
with a full queue equals the same proposals in runs that queue few (batches),
at mode numbers on both sides of each form's line.

Both forms evaluate in FP64 and round to FP32, so the integer statistics and the
copies are equal, and a sum of u(0)^p may differ by a rounding of a few terms:
an FP32 ulp of the largest for each."""
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


def _same(a, b, K):
    for p, q in zip(a, b):
        for f in ("n_proposals", "n_accepted", "n_kept", "n_refined", "n_near_threshold", "n_fallback"):
            assert p[f] == q[f], f
        assert np.array_equal(p["hist"], q["hist"]) and np.array_equal(p["exceed"], q["exceed"])
        top = np.sqrt(2 * K / np.pi)
        for e in range(4):  # a hundred terms off by one FP32 ulp
            assert abs(p["sum_u0"][e] - q["sum_u0"][e]) <= 100 * 2.0**-23 * top ** (e + 1)
        assert np.all(np.abs(p["spectrum"] - q["spectrum"]) <= 100 * 2.0**-23)


@pytest.mark.parametrize("K", [3, 8, 9, 14, 15, 17, 20, 21, 33, 34, 35, 41])
def test_full_queue_equals_short_queues(T, K):
    # beta' = 0: every proposal has weight 1, 63 % of them get a copy and are queued
    n, pts = 1 << 16, [T.make_point(0.0, 1.0, 0.0, T.PROPOSAL_UNIFORM, point_id=p, logM=0.0) for p in range(3)]
    S = T.Sampler(K, pts, sir=True, sample_capacity=1 << 18)
    S.run(n, 5)  # 124,000 queued
    full, rec = S.stats(), S.samples(1 << 18)
    S.reset()
    for i in range(8):  # 15,500 queued
        S.run(n // 8, 5)
    short, part = S.stats(), S.samples(1 << 18)
    S.close()
    assert sum(s["n_refined"] for s in full) > 110_000 and all(s["n_dropped"] == 0 for s in full)
    _same(full, short, K)
    a, b = (np.lexsort((r["idx"], r["point"])) for r in (rec, part))
    for f in ("point", "idx", "copies"):
        assert np.array_equal(rec[f][a], part[f][b]), f
    for f in ("H2", "u0", "xhat"):
        assert np.all(np.abs(rec[f][a] - part[f][b]) <= 2.0**-22 * np.abs(part[f][b])), f
    # T is a sum of O(1) terms in FP64
    assert np.all(np.abs(rec["H3"][a] - part["H3"][b]) <= 2.0**-22 * np.abs(part["H3"][b]) + 1e-12)


@pytest.mark.parametrize("K,cap", [(7, 16), (16, 1000), (32, 30_000), (64, 5)])
def test_sir_ring_smaller_than_the_queue(T, K, cap):
    got = []
    for c in (1 << 16, cap):
        S = T.Sampler(K, [T.make_point(0.0, 1.0, 0.0, T.PROPOSAL_UNIFORM, point_id=p, logM=0.0) for p in range(4)],
                      sir=True, sample_capacity=c)
        S.run(1 << 14, 9)  # 41,000 queued
        got.append((S.stats(), S.samples(1 << 16)))
        S.close()
    (big, rec), (small, part) = got
    _same(big, small, K)
    assert sum(s["n_dropped"] for s in big) == 0
    assert sum(s["n_dropped"] for s in small) == sum(s["n_kept"] for s in small) - cap
    assert len(part["idx"]) == cap and all(0 <= s["n_dropped"] <= s["n_kept"] for s in small)
    want = {(int(p), int(i)): int(k) for p, i, k in zip(rec["point"], rec["idx"], rec["copies"])}
    have = {(int(p), int(i)): int(k) for p, i, k in zip(part["point"], part["idx"], part["copies"])}
    assert len(have) == cap and all(want[k] == v for k, v in have.items())
