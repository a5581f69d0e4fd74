"""A point whose envelope search fails (cH overflows: no finite log f/g) answers
that, whatever else is wrong with the handle."""
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


def _code(T, pt, **opt):
    with pytest.raises(T.TkdvError) as e:
        T.Sampler(8, [T.make_point(2.0, 1.0, 1.0), pt], **opt)
    return str(e.value)


def test_envelope_error_comes_first(T):
    bad = T.make_point(1e200, 1.0, 1e200, T.PROPOSAL_UNIFORM)
    alone = _code(T, bad, sample_capacity=16)
    assert "ENVELOPE" in alone
    assert _code(T, bad, sample_capacity=1 << 44) == alone  # a ring that no memory holds
    assert "OOM" in _code(T, T.make_point(2.0, 1.0, 1.0), sample_capacity=1 << 44)
