"""What the host clears and copies keeps its place among the runs of a handle
that has a stream of its own, with work pending on the legacy default stream
(the one torch uses), which does not hold the handle's stream back."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, SEED, K = 300_001, 11, 9


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_16952_gb300 import _build
    _build.build()
    import paper_2411_16952_gb300 as T
    return torch, T


def _sampler(T, form):
    return T.Sampler(K, [T.make_point(20.0, 1.0, 20.0), T.make_point(20.0, 1.0, 10.0)], h3_mode=form,
                     sample_capacity=1 << 12)


def _result(S):
    st = S.stats()
    keys = ("n_proposals", "n_accepted", "n_near_threshold", "n_refined", "n_dropped", "n_fallback")
    return [np.array([[s[k] for k in keys] for s in st])] + [np.array([s[k] for s in st])
                                                              for k in ("hist", "sum_u0", "spectrum")]


def _busy(torch):
    torch.cuda._sleep(100_000_000)  # about 50 ms on the legacy stream


@pytest.mark.parametrize("form", [0, 1])
def test_reset_comes_before_the_next_run(env, form):
    torch, T = env
    S = _sampler(T, form)
    S.run(N, SEED)
    ref = _result(S)
    assert ref[0][:, 1].min() > 10
    for _ in range(3):
        _busy(torch)
        S.reset()
        S.run(N, SEED)
        for a, b in zip(ref, _result(S)):
            assert np.array_equal(a, b)
    S.close()


@pytest.mark.parametrize("form", [0, 1])
def test_a_new_handle_is_initialised_before_its_first_run(env, form):
    torch, T = env
    ref = None
    for busy in (False, True, True):
        if busy:
            _busy(torch)
        S = _sampler(T, form)
        S.run(N, SEED)
        got = _result(S)
        S.close()
        ref = ref or got
        for a, b in zip(ref, got):
            assert np.array_equal(a, b)


def test_records_copied_on_the_device_are_those_of_the_finished_run(env):
    torch, T = env
    # every proposal is accepted (beta' = 0, uniform): both runs fill the ring
    cap, K = 1 << 20, 64
    S = T.Sampler(K, [T.make_point(0.0, 1.0, 0.0, T.PROPOSAL_UNIFORM, logM=0.0)], sample_capacity=cap)
    buf = torch.zeros(cap * T.tkdv_record_bytes(K), dtype=torch.uint8, device="cuda")
    want = torch.zeros_like(buf)
    for seed in (1, 2, 3):
        S.reset()
        S.run(cap, seed)
        S.sync()
        assert S.samples(cap, device_dst=want) == cap
        torch.cuda.synchronize()
        assert S.samples(cap, device_dst=buf) == cap
        S.reset()
        S.run(cap, seed + 100)  # while the copy of 570 MB is on its way
        S.sync()
        torch.cuda.synchronize()
        assert torch.equal(buf, want)
    S.close()
