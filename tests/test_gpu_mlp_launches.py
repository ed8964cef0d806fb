"""Training over more steps than one launch takes (4096): moments, bias
corrections and the loss go from one launch to the next, so the parameters are
those of the same steps in several calls, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("epochs,parts", [(129, 129), (260, 5), (128, 2)])
def test_launch_boundary(epochs, parts):
    from paper_1612_08091_gb300.qsim import MLP

    r = np.random.default_rng(epochs)
    n, batch = 64, 2  # 32 steps an epoch: 4128, 8320 and 4096 steps
    X = r.uniform(0.0, 1.0, (n, 16)).astype(np.float32)
    y = (X[:, 0] - 2.0 * X[:, 5] + 0.1 * r.standard_normal(n)).astype(np.float32)
    whole, split = MLP(hidden=32, seed=3), MLP(hidden=32, seed=3)
    loss = whole.train(X, y, epochs=epochs, batch=batch, lr=1e-3)
    for _ in range(parts):
        last = split.train(X, y, epochs=epochs // parts, batch=batch, lr=1e-3)
    np.testing.assert_array_equal(whole.params, split.params)
    assert loss == last
