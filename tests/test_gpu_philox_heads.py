"""The Philox blocks from a chunk's table of heads: runs whose range crosses a
multiple of 2^32 inside a chunk (the table holds for one upper half of the
index), at odd mode numbers and with a key and a point id that use all bits,
against the launch variants that make their blocks from the counter.  Records
and statistics are equal bit for bit."""
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


@pytest.mark.parametrize("K,mode,variants", [(9, 0, (0, 2, 5)), (16, 0, (0, 2, 5)), (17, 0, (1, 2, 5)),
                                             (32, 0, (4, 2, 5)), (13, 1, (1, 0)), (32, 1, (2, 0, 1))])
def test_heads_equal_counter_blocks(T, K, mode, variants):
    pts = [T.make_point(20.0, 1.0, 20.0, T.PROPOSAL_PAPER, point_id=0xFEDCBA98),
           T.make_point(20.0, 1.0, 10.0, T.PROPOSAL_UNIFORM, point_id=7)]
    ref = None
    for v in variants:
        S = T.Sampler(K, pts, h3_mode=mode, sample_capacity=1 << 18)
        S.set_launch(v)
        for lo in (0x1_0000_0000 - 5001, 0xFFFF_FFFF_0000_0000 - 77, 0x7_0000_0000 - 1):
            S.run_ranges([lo, lo + 3], [40_001, 12_345], 0x89ABCDEF_FEDCBA98)
        st, rec = S.stats(), S.samples(1 << 18)
        S.close()
        o = np.lexsort((rec["idx"], rec["point"]))
        got = [rec[f][o] for f in ("point", "idx", "u0", "xhat", "H2")]
        got += [np.array([[s[f] for f in ("n_proposals", "n_accepted", "n_refined", "n_near_threshold")] for s in st]),
                np.array([s["spectrum"] for s in st]), np.array([s["sum_u0"] for s in st])]
        assert len(got[0]) > 500
        if ref is None:
            ref = got
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), v
