"""Surrogate training and forward kernels at the edges of their tiles: mini-batches
around the 16-row tile and the 128-row chunk against the FP64 network oracle (the
tolerance of tests/test_gpu_surrogate.py, for its reason), and the splits that
must not change a value (members together or alone, mini-batches in one launch or many)."""
import numpy as np
import pytest

from oracle import mlp
from paper_2207_09431_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-3


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_09431_gb300 import lbm as _lbm

    _lbm.load_library()
    return _lbm


def relerr(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-30))


@pytest.mark.parametrize("rows", [2, 15, 16, 17, 112, 127, 128, 129, 255, 257, 384])
def test_gradients_at_tile_edges(lbm, rows):
    w = inputs.mlp_init(2, seed=21)
    net = lbm.Surrogate(w, max_batch=384, max_rows=384)
    rng = np.random.default_rng(rows)
    X, T = rng.normal(size=(rows, 5)), rng.normal(size=(rows, 2))
    Y, loss, g = net.forward_backward(1, X, T)
    params = inputs.mlp_unflatten(w[1])
    Yo, cache = mlp.forward(params, X)
    assert relerr(Y, Yo) < TOL
    assert abs(loss - mlp.loss(Yo, T)) <= TOL * mlp.loss(Yo, T)
    go = mlp.backward(params, cache, Yo, T)
    for got, want in zip(inputs.mlp_unflatten(g), go):
        assert relerr(got[0], want[0]) < TOL and relerr(got[1], want[1]) < TOL
    assert np.array_equal(net.forward_backward(1, X)[0], Y)  # the forward kernel's sums run in the same order


@pytest.mark.parametrize("rows,batch", [(40, 1), (50, 17), (300, 130), (256, 256)])
def test_splits_change_no_value(lbm, rows, batch):
    rng = np.random.default_rng(batch)
    X, Y = rng.normal(size=(rows, 5)), rng.normal(size=(rows, 2))
    w = inputs.mlp_init(16, seed=22)
    together = lbm.Surrogate(w, max_batch=batch, max_rows=rows)  # the least scratch: many launches
    alone = lbm.Surrogate(w[:1], max_batch=512, max_rows=rows)
    for seed in (0, 1):  # the second call goes on from the first's moments
        together.train(X, Y, epochs=3, batch=batch, lr=2e-3, seed=seed)
        alone.train(X, Y, epochs=3, batch=batch, lr=2e-3, seed=seed)
        assert np.array_equal(together.weights(0), alone.weights(0))
    assert not np.array_equal(together.weights(1), w[1].astype(np.float32))
    mean, spread, _ = together.predict(X[:batch])
    y = np.stack([together.forward_backward(m, (X[:batch] - X.mean(0)) / X.std(0))[0] for m in range(16)])
    y = y * Y.std(0) + Y.mean(0)
    # the raw outputs here start from inputs normalised in another order (FP32 rounding of the
    # normalised inputs may differ by one unit, BF16 operands by one in rare places)
    assert relerr(mean, y.mean(0)) < TOL and spread.shape == (batch, 2)
