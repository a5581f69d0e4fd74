"""Full chunks of the grid form that cross a multiple of 2^32 with every
proposal accepted: a warp then holds the accepted draws of 65 tiles.  The run
that crosses inside a chunk equals the same proposals in two ranges that end
and begin at the multiple, sum for sum."""
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


@pytest.mark.parametrize("K,before", [(3, 100), (3, 64), (17, 64), (33, 8191 - 128 * 3)])
def test_every_draw_of_a_split_chunk_is_kept_once(T, K, before):
    # beta' = 0 under the uniform proposal: log f/(Mg) = 0, every u < 1 accepts
    S = T.Sampler(K, [T.make_point(0.0, 1.0, 0.0, T.PROPOSAL_UNIFORM, logM=0.0)], h3_mode=T.H3_GRID_BF16X3,
                  sample_capacity=16)
    cfg = S.launch_config()
    workers = cfg["ctas"] * (cfg["threads"] // 128)
    n = 8 * workers * 8192 - 5  # full chunks, the multiple of 2^32 in the first
    got = []
    for ranges in ([(2**32 - before, n)], [(2**32 - before, before), (2**32, n - before)]):
        S.reset()
        for lo, cnt in ranges:
            S.run_ranges([lo], [cnt], 7)
            if cnt == n:
                assert S.launch_config()["chunk"] == 8192
        got.append(S.stats()[0])
    S.close()
    for st in got:
        assert st["n_proposals"] == n and st["n_accepted"] == n and st["n_dropped"] == n - 16
        assert int(st["hist"].sum()) == n
        assert abs(st["spectrum"].sum() / n - 1.0) < 1e-5  # sum_k s_k = 1 in FP32, K terms of a few 2^-24
    for f in ("hist", "exceed", "sum_u0", "spectrum"):
        assert np.array_equal(got[0][f], got[1][f]), f
