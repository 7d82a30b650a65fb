"""Expired waits of the surrogate network's tensor-core kernels, without a GPU fault.

With a wait limit of 0 polls every bounded mbarrier wait runs out. The call that started the work says
so, training leaves the parameters and moments of the last complete step, and the network goes on.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TIMEOUT = -6


def _expired(call):
    from paper_2412_10167_gb300 import mw3
    with pytest.raises(mw3.MW3Error) as e:
        call()
    assert e.value.code == TIMEOUT


@pytest.mark.parametrize("width,depth,rows", [(96, 2, 40), (128, 3, 700), (256, 2, 33), (200, 4, 9000)])
def test_expired_wait_leaves_the_network_usable(width, depth, rows):
    from paper_2412_10167_gb300 import mw3
    g = np.random.default_rng(21)
    X = g.standard_normal((rows, 4)).astype(np.float32)
    y = np.sin(2 * X[:, 0]).astype(np.float32)
    nets = [mw3.MLP(n_in=4, width=width, depth=depth, seed=22) for _ in range(2)]
    for net in nets:
        net.train(X, y, 1, batch=32, lr=1e-2, seed=1)
    a, b = nets
    p, out, (loss, grad) = a.get_params(), a.forward(X), a.loss_grad(X, y)
    a.set_wait_limit(0)
    _expired(lambda: a.forward(X))
    _expired(lambda: a.loss_grad(X, y))
    _expired(lambda: a.train(X, y, 2, batch=32, lr=1e-2, seed=2))
    a.set_wait_limit(1 << 22)
    assert np.array_equal(a.get_params(), p)
    assert np.array_equal(a.forward(X), out)
    l2, g2 = a.loss_grad(X, y)
    assert l2 == loss and np.array_equal(g2, grad)
    # moments and step count as well: the next epoch is that of a network without the failure
    assert a.train(X, y, 1, batch=32, lr=1e-2, seed=3) == b.train(X, y, 1, batch=32, lr=1e-2, seed=3)
    assert np.array_equal(a.get_params(), b.get_params())
    for net in nets:
        net.close()


def test_wait_limit_range():
    from paper_2412_10167_gb300 import mw3
    net = mw3.MLP(n_in=2, width=8, depth=1, seed=1)
    for polls in (-1, (1 << 22) + 1):
        with pytest.raises(mw3.MW3Error):
            net.set_wait_limit(polls)
    net.close()
