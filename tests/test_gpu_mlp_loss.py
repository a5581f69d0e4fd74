"""The loss kernel of the network's training (4, 8 or 16 lanes to a row) at
mode numbers around its column layouts and row counts around a warp's 32 rows
and the blocks of a point, one to many points, against FP64 backpropagation
with the same BF16 weights.  Bounds: those of test_gpu_learned.py's gradient
test, whose sums are the same FP32 ones."""
import numpy as np
import pytest

from oracle import mlp as OM

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


@pytest.mark.parametrize("Ks,rows", [((1,), (1,)), ((4, 3), (31, 33)), ((5,), (257,)), ((16, 15), (32, 1)),
                                     ((17, 2, 32), (100, 8191, 4)), ((33,), (1000,)), ((64, 61), (65, 3000)),
                                     ((32,) * 24, tuple(range(1, 25)))])
@pytest.mark.parametrize("tau", [0.0, 0.5])
def test_loss_and_gradient(T, Ks, rows, tau):
    g = np.random.default_rng(len(rows) + sum(rows))
    P = len(Ks)
    feats = g.uniform(-1, 1, (P, 4)).astype(np.float32).astype(np.float64)
    wp = [g.uniform(1, 3, K).astype(np.float32).astype(np.float64) for K in Ks]
    s = [g.dirichlet(np.ones(K), n).astype(np.float32).astype(np.float64) for K, n in zip(Ks, rows)]
    z = [g.normal(0, 1.5, n).astype(np.float32).astype(np.float64) for n in rows]
    m = T.tkdv_mlp_create(0)
    T.tkdv_mlp_set_params(m, (0.15 * g.standard_normal(T.MLP_NPARAM)).astype(np.float32))
    _, w = T.tkdv_mlp_get_params(m)
    T.tkdv_mlp_set_data(m, list(Ks), feats, wp, s, z)
    loss, grad = T.tkdv_mlp_step(m, lr=1e-3, tau=tau, update=False, want_grad=True)
    again, grad2 = T.tkdv_mlp_step(m, lr=1e-3, tau=tau, update=True, want_grad=True)
    assert loss == again and np.array_equal(grad, grad2)
    moved = T.tkdv_mlp_step(m, lr=1e-3, tau=tau, update=False)  # the step before wrote the weights this one reads
    T.tkdv_mlp_destroy(m)
    th, o = {}, 0
    w = w.astype(np.float64)
    for name, shape in (("W1", (64, 4)), ("b1", (64,)), ("W2", (64, 64)), ("b2", (64,)), ("W3", (64, 64)), ("b3", (64,))):
        k = int(np.prod(shape))
        th[name] = w[o:o + k].reshape(shape)
        o += k
    J, gr = OM.loss_and_grad(th, feats, list(Ks), wp, s, z, None if tau <= 0 else tau)
    ref = np.concatenate([gr[n].ravel() for n in ("W1", "b1", "W2", "b2", "W3", "b3")])
    assert abs(loss - J) <= 1e-4 * (1 + abs(J))
    assert np.max(np.abs(grad - ref)) <= 2e-3 * (np.max(np.abs(ref)) + 1e-6)
    if np.max(np.abs(ref)) > 1e-3:
        assert moved < loss
