"""An error that an earlier CUDA call of the thread left behind (here a ring that
no memory holds) does not make the next handle, its fields' maxima or its extreme
field fail."""
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


def _fail(T):
    with pytest.raises(T.TkdvError):
        T.Sampler(8, [T.make_point(2.0, 1.0, 1.0, logM=3.0)], sample_capacity=1 << 44)


def test_calls_after_a_failed_allocation(T):
    _fail(T)
    S = T.Sampler(8, [T.make_point(2.0, 1.0, 1.0)], sample_capacity=1 << 14)
    S.run(1 << 14, 3)
    _fail(T)
    umax, _ = S.field_maxima(1 << 14)
    _fail(T)
    ev = S.extreme_field(m=len(umax))
    assert ev["umax"] == np.max(umax)
    _fail(T)
    st = T.sampler_batch_run([T.make_point(2.0, 1.0, 1.0)], T.make_options(8, sample_capacity=16), [1 << 14], 3)
    assert st[0]["n_accepted"] == S.stats()[0]["n_accepted"] == len(umax)
    S.close()


def test_training_step_after_a_failed_allocation(T):
    K, n, rng = 8, 512, np.random.default_rng(1)
    s = rng.random((n, K)).astype(np.float32)
    s /= s.sum(1, keepdims=True)
    w0 = (0.1 * rng.standard_normal(T.MLP_NPARAM)).astype(np.float32)
    got = []
    for fail in (False, True):
        m = T.tkdv_mlp_create(0)
        T.tkdv_mlp_set_params(m, w0)
        T.tkdv_mlp_set_data(m, [K], [T.tkdv_mlp_features(K, 2.0, 1.0, 1.0)], [np.ones(K)], [s])
        for _ in range(3):
            if fail:
                _fail(T)
            loss, grad = T.tkdv_mlp_step(m, lr=1e-2, tau=1.0, update=True, want_grad=True)
        got.append([np.array(loss), grad, *T.tkdv_mlp_get_params(m)])
        T.tkdv_mlp_destroy(m)
    for a, b in zip(*got):
        assert np.array_equal(a, b)
