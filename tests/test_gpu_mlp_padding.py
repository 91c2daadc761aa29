"""Tensor-core inference with hidden widths that are padded to multiples of 16: an activation that overflows to infinity
stays one in the outputs (a padded column is zero, not zero weights times infinity), and the other rows of its tile are
as without it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden", [24, 40, 250])
@pytest.mark.parametrize("n", [3, 40000])
def test_infinite_activation(hidden, n):
    from paper_1009_2727_gb300.surrogate import MLP
    widths = [2, hidden, hidden, 2]
    rng = np.random.default_rng(5)
    w1, w2, w3 = np.zeros((hidden, 2)), np.ones((hidden, hidden)) / hidden, np.ones((2, hidden)) / hidden
    w1[:, 1] = 1.0
    w1[0] = (1e30, 1.0)     # overflows for the first input 1e20, unit 0 alone
    w3[1] = -w3[1]
    net = MLP(widths, seed=1)
    net.set_params(np.concatenate([v.reshape(-1) for w, b in ((w1, hidden), (w2, hidden), (w3, 2)) for v in (w, np.zeros(b))]))
    x = np.zeros((n, 2), dtype=np.float32)
    x[:, 1] = rng.uniform(0.5, 2.0, n)
    plain = net.forward(x)
    assert np.isfinite(plain).all()
    big = x.copy()
    rows = np.arange(0, n, 2)
    big[rows, 0] = 1e20
    y = net.forward(big)
    assert (y[rows, 0] == np.inf).all() and (y[rows, 1] == -np.inf).all()
    rest = np.arange(1, n, 2)
    assert np.array_equal(y[rest], plain[rest])
    net.close()
