"""The fused network kernels at the edges of their tiles: 8-sample training
tiles, inference tiles of 16 to 80 samples, 64-sample gradient chunks."""
import numpy as np
import pytest

from oracle import mlp
from paper_2504_09024_gb300 import lbm

pytestmark = pytest.mark.gpu


def inputs(n, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(-1.0, 1.0, (n, 5)).astype(np.float32),
            rng.uniform(0.0, 0.4, n).astype(np.float32),
            (rng.uniform(size=n) < 0.4).astype(np.float32))


# one wave of 152 blocks takes 2432, 4864, 7296, 9728 and 12160 samples with 1
# to 5 samples a thread; beyond that blocks walk several tiles
@pytest.mark.parametrize("n", [1, 15, 17, 2432, 2433, 4865, 7297, 9729, 12161, 30011])
def test_predictions_do_not_depend_on_the_tiling(n):
    """A sample's outputs are one fixed chain of operations: the same bits in
    any batch, here against batches of 8."""
    net = lbm.Surrogate(seed=5)
    X, _, _ = inputs(n, n)
    D, z = net.predict(X)
    rng = np.random.default_rng(1)
    at = np.unique(np.concatenate([rng.integers(0, n, 24), [0, n - 1, n // 2]]))
    for a in range(0, len(at), 8):
        k = at[a:a + 8]
        d8, z8 = net.predict(X[k])
        np.testing.assert_array_equal(D[k], d8)
        np.testing.assert_array_equal(z[k], z8)
    net.close()


@pytest.mark.parametrize("n", [1, 8, 9, 63, 64, 65, 193, 1217])
def test_gradients_at_tile_edges(n):
    """Against the FP64 reference.  FP32
    chains of at most 1217 terms: 1e-4 relative covers 1217 roundings of 6e-8
    that all add up, through five layers."""
    params = mlp.init_params(seed=9)
    net = lbm.Surrogate(seed=1)
    net.set_params(params)
    X, yD, yB = inputs(n, 100 + n)
    got, loss = net.grad(X, yD, yB)
    X64, D64 = X.astype(np.float64), yD.astype(np.float64)
    out, cache = mlp.forward(params, X64)
    ref = mlp.backward(params, cache, out, D64, yB.astype(np.float64))
    for (gW, gb), (rW, rb) in zip(got, ref):
        assert np.linalg.norm(gW - rW) <= 1e-4 * np.linalg.norm(rW)
        assert np.linalg.norm(gb - rb) <= 1e-4 * np.linalg.norm(rb)
    assert abs(loss - mlp.loss(out, D64, yB)) <= 1e-5 * abs(loss)
    net.close()


def test_training_twice_is_training_through():
    """Two calls of 3 and 5 epochs leave the bits of one call of 8."""
    X, yD, yB = inputs(130, 3)
    a, b = lbm.Surrogate(seed=2), lbm.Surrogate(seed=2)
    a.train(X, yD, yB, epochs=8, lr=2e-3)
    b.train(X, yD, yB, epochs=3, lr=2e-3)
    b.train(X, yD, yB, epochs=5, lr=2e-3)
    for (W, c), (W2, c2) in zip(a.get_params(), b.get_params()):
        np.testing.assert_array_equal(W, W2)
        np.testing.assert_array_equal(c, c2)
    a.close()
    b.close()
