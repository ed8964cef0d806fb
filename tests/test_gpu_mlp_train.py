"""The many-steps training kernel of the cost model (up to 64 hidden units,
a multiple of 4) and the per-layer path of the other widths: one Adam step
from the per-layer gradient, and the loss of an epoch with a partial last
batch, at the edges of the kernel's row, column and chunk splits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1612_08091_gb300.qsim import MLP

    return MLP


def data(n, seed):
    r = np.random.default_rng(seed)
    X = r.uniform(-1, 1, (n, 16)).astype(np.float32)
    return X, (X[:, 0] - X[:, 3] * X[:, 5]).astype(np.float32)


def adam1(p, g, lr):
    """The first Adam step in FP64 from an FP32 gradient."""
    g = g.astype(np.float64)
    m, v = (1 - float(np.float32(0.9))) * g, (1 - float(np.float32(0.999))) * g * g
    c1, c2 = 1 - float(np.float32(0.9)), 1 - float(np.float32(0.999))
    return p - lr * (m / c1) / (np.sqrt(v / c2) + 1e-8)


@pytest.mark.parametrize("hidden", [4, 12, 16, 32, 48, 60, 64, 30, 68])
@pytest.mark.parametrize("n", [1, 7, 8, 33, 256, 300])
def test_one_step_is_the_gradient_step(mlp, hidden, n):
    X, T = data(n, hidden * 1000 + n)
    net = mlp(hidden=hidden, seed=3)
    p0 = net.params
    g, loss0 = net.gradient(X, T)
    loss = net.train(X, T, epochs=1, batch=n, lr=1e-3)
    want = adam1(p0.astype(np.float64), g, float(np.float32(1e-3)))
    # about ten FP32 roundings of an update of at most lr, and one of p; below
    # |g| = 1e-4 the epsilon of the denominator joins them
    tol = 2.0 ** -24 * np.maximum(np.abs(p0), 1.0) + 1e-3 * 1e-4
    assert np.all(np.abs(net.params - want) <= tol)
    assert abs(loss - loss0) <= 1e-6 * max(1.0, loss0)
    net.close()


@pytest.mark.parametrize("hidden", [32, 64])
def test_partial_batches_and_the_epoch_loss(mlp, hidden):
    n, batch = 300, 64  # 5 steps, the last of 44 samples
    X, T = data(n, hidden)
    a, b = mlp(hidden=hidden, seed=5), mlp(hidden=hidden, seed=5)
    loss = a.train(X, T, epochs=2, batch=batch, lr=1e-3)
    # the same two epochs, each epoch's loss from a run of its own
    first = b.train(X, T, epochs=1, batch=batch, lr=1e-3)
    second = b.train(X, T, epochs=1, batch=batch, lr=1e-3)
    np.testing.assert_array_equal(a.params, b.params)
    assert loss == second and second < first
    a.close()
    b.close()
