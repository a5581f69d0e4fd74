"""The envelope search on the device (real amplitudes, one warp per start)
against tkdv_log_M, the host's search over the whole sphere: every proposal
kind, both signs of C3/C2 and zero, beta' from 0 to near the largest with an
alpha*, mode numbers at the edges of the kernel's lane layouts.  Both stop at
the last bits of log f/g, a maximum where the value is flat: 1e-10 relative."""
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


@pytest.mark.parametrize("K,n", [(1, 6), (2, 12), (3, 12), (4, 12), (7, 12), (16, 24), (31, 12), (32, 24), (33, 6),
                                 (48, 6), (63, 3), (64, 3), (65, 2), (100, 2), (128, 2)])
def test_device_envelope_equals_host_search(T, K, n):
    g = np.random.default_rng(K)
    top = 0.95 * K * K * np.sum(1.0 / np.arange(1, K + 1) ** 2)
    pts, own = [], []
    for i in range(n):
        prop = (T.PROPOSAL_PAPER, T.PROPOSAL_UNIFORM, T.PROPOSAL_LEARNED)[i % 3]
        beta = 0.0 if i == 4 else float(np.exp(g.uniform(np.log(0.05), np.log(top))))
        lam = 0.0 if i == 5 else float(10.0 ** g.uniform(0, 4.5)) * (-1 if i % 4 == 3 else 1)
        E0 = float(g.uniform(0.5, 2.0))
        corr = 0.3 * np.cos(0.4 * np.arange(1, K + 1)) if prop == T.PROPOSAL_LEARNED else None
        pts.append(T.make_point(beta, E0, lam / max(beta, 1.0), prop, point_id=i, log_var_correction=corr))
        own.append((beta, E0, lam / max(beta, 1.0), prop))
    pts.append(T.make_point(1.0 if K > 1 else 0.5, 1.0, 0.0, T.PROPOSAL_PAPER, logM=3.25))  # keeps its own
    S = T.Sampler(K, pts, sample_capacity=16)
    info = [S.point_info(p) for p in range(n + 1)]
    S.close()
    assert info[n][1] == 3.25
    for (beta, E0, r, prop), (_, lm, s2) in zip(own, info):
        ref = T.tkdv_log_M(K, beta, E0, r, None if prop == T.PROPOSAL_UNIFORM else s2)
        assert abs(lm - ref) <= 1e-10 * (1 + abs(ref)), (K, beta, E0, r, prop, lm, ref)
