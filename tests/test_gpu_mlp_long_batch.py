"""Gradient of a long batch against the FP64 oracle.

Its sums run over the batch; rounded to nearest their error does not grow with it, while an
accumulator that truncates shifts every term the same way. The error left is that of the activations
and of the loss gradient, a few 2^-24 each, which the network amplifies up to ten times: 1e-6 of
the gradient's norm at any number of rows."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


def _bf16(x):
    u = np.asarray(x, dtype=np.float32).view(np.uint32).astype(np.uint64)
    return ((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32).astype(np.float64)


@pytest.mark.parametrize("width,depth,rows", [(256, 3, 120000), (96, 2, 100001)])
def test_gradient_error_does_not_grow_with_the_batch(width, depth, rows):
    from paper_2412_10167_gb300 import mw3
    net = mw3.MLP(n_in=4, width=width, depth=depth, seed=12)
    net.set_params(_bf16(net.get_params()))
    p = net.get_params()
    g = np.random.default_rng(13)
    X = g.standard_normal((rows, 4)).astype(np.float32)
    y = (np.sin(2 * X[:, 0]) + 0.1 * X.sum(axis=1)).astype(np.float32)
    params = [[W.astype(float).copy(), b.astype(float).copy()] for W, b in net.unflatten(p)]
    _, ref = omlp.loss_and_grads(params, X.astype(float), y.astype(float))
    ref = np.concatenate([np.concatenate([a.ravel(), b]) for a, b in ref])
    _, grad = net.loss_grad(X, y)
    net.close()
    assert np.linalg.norm(grad - ref) <= 1e-6 * np.linalg.norm(ref)
