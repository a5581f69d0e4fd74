"""The FP64 pass of up to 64 modes (a warp takes a batch of queued proposals,
the modes and triads of each spread over a segment of its lanes) against the
oracle.  SIR runs send every proposal that may get a copy through it, so the
queue holds from one item (fewer than the warps: batches of one segment group)
to tens of thousands (batches of 32), at the mode numbers where the lane
segments change and at their neighbours.

Both sides evaluate in FP64 and the kernel rounds its results to FP32 (2^-24),
with the FP32 scale of u(0) and H3 (another 2^-24): relative 2^-22."""
import numpy as np
import pytest

import oracle as O

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


@pytest.mark.parametrize("n", [3, 701, 1 << 15])
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 32, 33, 47, 63, 64])
def test_fp64_pass_matches_oracle(T, K, n):
    prop, tprop = (O.UNIFORM, T.PROPOSAL_UNIFORM) if K % 3 == 0 else (O.PAPER, T.PROPOSAL_PAPER)
    bp, E0, pid, seed = min(20.0, 0.4 * K * K), 1.0, 3, 11 + K
    r = K**1.5 / bp
    pt = O.make_point(K, E0, bp, r, prop)
    # any log M gives a valid SIR run: here the largest weights are of order one, so that many proposals are queued
    pt.logM = float(np.max(O.replay(pt, seed, pid, np.arange(2048, dtype=np.uint64))["logfg"]))
    S = T.Sampler(K, [T.make_point(bp, E0, r, tprop, point_id=pid, logM=pt.logM, sir_c=0.7)], sir=True,
                  sample_capacity=n)
    S.run_ranges([0], [n], seed)
    st = S.stats()[0]
    rec = S.samples(n)
    S.close()
    ost, kept = O.run_sir(pt, seed, pid, 0, n, 0.7, cap=n)
    a, b = np.argsort(rec["idx"]), np.argsort(kept["idx"])
    assert np.array_equal(rec["idx"][a], kept["idx"][b]) and np.array_equal(rec["copies"][a], kept["copies"][b])
    assert st["n_kept"] == len(a) and st["n_accepted"] == kept["copies"].sum() and st["n_refined"] >= len(a)
    for f in ("H2", "H3", "u0", "xhat"):
        g, o = rec[f][a].astype(np.float64), kept[f][b].astype(np.float64)
        assert np.all(np.abs(g - o) <= 2.0**-22 * np.abs(o) + 1e-10), f
    spec = (kept["copies"][b][:, None] * (kept["xhat"][b][:, :K] ** 2 + kept["xhat"][b][:, K:] ** 2)).sum(0)
    assert np.all(np.abs(st["spectrum"][:K] - spec) <= 2.0**-21 * spec + 2.0**-28 * n)
