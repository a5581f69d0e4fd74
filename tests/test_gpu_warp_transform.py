"""H3 of the warp form (65..128 modes) by the fast transform on 384 points:
against the oracle's double sum in FP64, at the mode numbers where its columns
begin and end (k = 120 + k1 <= 128, k >= 256 standing for k - 384) and at K =
128, whose top mode aliases; batches with one to four proposals; indices on
both sides of 2^32, where the Philox words shared by a run change.

Bound: 75 2^-24 sqrt(K) on T for the transform (sampler_k128.cu) and as much
again for the FP32 draw (sin and cos within 2^-21.4 of the amplitude, the
radius within 2^-22: below 8 2^-24 per component, three times that in T with
|T| <= sqrt(K)), H3 = 2 pi (E0/2pi)^{3/2} T."""
import math

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


@pytest.mark.parametrize("K", [65, 66, 71, 72, 73, 96, 97, 119, 120, 121, 127, 128])
def test_transform_matches_oracle(T, K):
    prop, tprop = (O.UNIFORM, T.PROPOSAL_UNIFORM) if K % 2 else (O.PAPER, T.PROPOSAL_PAPER)
    bp, E0, r, seed, pid = 30.0, 1.0, 100.0, 5, 9
    pt = O.make_point(K, E0, bp, r, prop)
    pt.logM = 300.0  # nothing near the threshold: every value from the FP32 path
    S = T.Sampler(K, [T.make_point(bp, E0, r, tprop, point_id=pid, logM=300.0)], sample_capacity=16)
    idx = np.concatenate([np.arange(1021), (1 << 32) - 514 + np.arange(1026)]).astype(np.uint64)
    g, o = S.replay(0, idx, seed), O.replay(pt, seed, pid, idx)
    S.close()
    fast = g["flags"] == 0
    assert fast.sum() > 2000
    h3s = 2 * math.pi * (E0 / (2 * math.pi)) ** 1.5
    assert np.all(np.abs(g["H3"] - o["H3"])[fast] <= h3s * math.sqrt(K) * 150 * 2.0**-24)
    assert np.all(np.abs(g["xhat"] - o["xhat"])[fast] <= 2e-6)
    for n in (1, 2, 3, 5):  # batches that are not full
        S2 = T.Sampler(K, [T.make_point(bp, E0, r, tprop, point_id=pid, logM=300.0)], sample_capacity=16)
        h = S2.replay(0, idx[:n], seed)
        S2.close()
        assert np.array_equal(h["H3"], g["H3"][:n]) and np.array_equal(h["xhat"], g["xhat"][:n])
