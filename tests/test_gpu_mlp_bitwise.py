"""The small-batch products sum in the order of the large tiles: their gradients are those of the tiled kernels bit for bit.
The same rows in a batch of more than 512 rows whose further rows have the network's own outputs as targets (zero gradient,
adding nothing): all gradients are 2^-k of the small batch's, k the ratio of the row counts, an exact factor."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [[6, 256, 256, 256, 4], [5, 33, 17, 3], [16, 264, 300, 20], [7, 9]])
@pytest.mark.parametrize("n", [1, 15, 64, 300, 512])
def test_gradient_of_the_tiles(widths, n):
    from paper_1009_2727_gb300.surrogate import MLP
    rng = np.random.default_rng(n)
    net = MLP(widths, seed=3)
    net.set_params(net.get_params() + rng.normal(0, 0.05, net.n_params).astype(np.float32))
    net.use_tensor_cores(False)
    k = 1
    while n << k <= 512:
        k += 1
    x = rng.normal(0, 1, (n << k, widths[0])).astype(np.float32)
    t = net.forward(x)                       # the tiled products
    _, zero = net.grad(x, t)                 # as the gradient's forward pass has them
    assert not zero.any()
    _, zero = net.grad(x[:n], t[:n])         # and the small batch's
    assert not zero.any()
    t[:n] += rng.normal(0, 1, (n, widths[-1])).astype(np.float32)
    small_loss, small = net.grad(x[:n], t[:n])
    large_loss, large = net.grad(x, t)
    assert np.array_equal(small, large * np.float32(1 << k))
    assert small_loss == pytest.approx(large_loss * (1 << k), rel=1e-5)
    net.close()
