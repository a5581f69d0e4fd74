"""The number of a point's fields where more of them are asked for than there are
records: nothing is selected."""
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


@pytest.mark.parametrize("kept", [1, 37, 4096])
def test_count_alone(T, kept):
    # m above the number of records: the fields of the point are only counted
    S = T.Sampler(4, [T.make_point(0.0, 1.0, 0.0, T.PROPOSAL_UNIFORM, logM=0.0) for _ in range(2)],
                  sample_capacity=8192)
    S.run_budgets([kept, 3], 5)
    for point, n in ((0, kept), (1, 3)):
        for m in (kept + 4, 1 << 62, (1 << 64) - 1):
            assert T.sampler_extreme_field(S.h, 4, point, m, 1 << 62) == (n, None)
    n, best = T.sampler_extreme_field(S.h, 4, 0, kept, 1 << 62)
    assert n == kept and best[0] < kept
    S.close()
