"""Batches whose activations pass through the network in several passes.

A batch that repeats its rows 1024 times has the loss and gradient of the rows themselves: every row's
values are the same up to the exact factor 2^-10 of the mean, only the sums are cut differently. The
targets keep the sums from cancelling, so that FP32 sums agree to a few 2^-24: 1e-6 of the norm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _data(rows, seed):
    g = np.random.default_rng(seed)
    X = g.standard_normal((rows, 4)).astype(np.float32)
    return X, (3.0 + 0.1 * np.sin(2 * X[:, 0])).astype(np.float32)


def test_batch_larger_than_the_memory_of_its_padded_activations():
    from paper_2412_10167_gb300 import mw3
    net = mw3.MLP(n_in=4, width=32, depth=16, seed=31)
    X, y = _data(12700, 32)                  # x 1024: 320 GB of activations padded to 128 neurons
    loss, grad = net.loss_grad(X, y)
    l2, g2 = net.loss_grad(np.tile(X, (1024, 1)), np.tile(y, 1024))
    net.close()
    assert abs(l2 - loss) <= 1e-12 * loss
    assert np.linalg.norm(g2 - grad) <= 1e-6 * np.linalg.norm(grad)


def test_training_step_of_several_passes():
    """The first step is lr times the gradient's sign, in one pass or two (400,000 shuffled rows)."""
    from paper_2412_10167_gb300 import mw3
    net = mw3.MLP(n_in=4, width=32, depth=16, seed=33)
    X, y = _data(400000, 34)
    p, (loss, g) = net.get_params(), net.loss_grad(X, y)
    assert abs(net.train(X, y, 1, batch=400000, lr=1e-3, seed=1) - loss) <= 1e-12 * loss
    q = net.get_params()
    net.close()
    big = np.abs(g) > 1e-4 * np.abs(g).max()
    assert np.max(np.abs((p - q)[big] - 1e-3 * np.sign(g[big]))) <= 2e-6
