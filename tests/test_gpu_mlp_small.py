"""Gradients and training of small batches (the 16 x 16 tiles and the fused gradient + AdamW launch) at the edges of the
tiles, the reduction slice and the row limit, against the FP64 oracle of the network.

Tolerances as in the other network tests (BF16 activations, unit roundoff 2^-9): 3e-2 relative L2 on the gradient,
2e-2 on the loss. A training step moves each parameter by lr (m / (sqrt(v) + eps) + wd p): from a zero state the first
step is lr sign(g), so after it every parameter with a gradient well above the rounding agrees with the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def bf16(a):
    u = np.ascontiguousarray(a, dtype=np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def rounded(p, widths):
    q, o = np.asarray(p, dtype=np.float64).copy(), 0
    for a, b in zip(widths[:-1], widths[1:]):
        q[o:o + a * b] = bf16(p[o:o + a * b])
        o += a * b + b
    return q


@pytest.mark.parametrize("widths,n", [
    ([6, 256, 256, 256, 4], 64), ([6, 256, 256, 256, 4], 512), ([6, 256, 256, 256, 4], 513), ([5, 33, 17, 3], 15),
    ([16, 264, 300, 20], 17), ([3, 1, 5], 1), ([7, 9], 33), ([8, 512, 8], 65)])
def test_small_batch_gradient(widths, n):
    from oracle import mlp as ref
    from paper_1009_2727_gb300.surrogate import MLP
    rng = np.random.default_rng(n)
    net = MLP(widths, seed=3)
    p = net.get_params() + rng.normal(0, 0.05, net.n_params).astype(np.float32)
    net.set_params(p)
    x, t = rng.normal(0, 1, (n, widths[0])), rng.normal(0, 1, (n, widths[-1]))
    loss_ref, g_ref = ref.loss_and_grad(rounded(p, widths), widths, bf16(x), t)
    for _ in range(2):   # a second pass over the same buffers
        loss, g = net.grad(x, t)
        assert loss == pytest.approx(loss_ref, rel=2e-2)
        assert np.linalg.norm(g - g_ref) <= 3e-2 * np.linalg.norm(g_ref)
    net.close()


@pytest.mark.parametrize("widths,n,batch", [([6, 256, 256, 256, 4], 64, 64), ([5, 33, 17, 3], 50, 50), ([7, 9], 16, 16)])
def test_small_batch_adamw_step(widths, n, batch):
    from oracle import mlp as ref
    from paper_1009_2727_gb300.surrogate import MLP
    rng = np.random.default_rng(5)
    net = MLP(widths, seed=4)
    p = net.get_params()
    x, t = rng.normal(0, 1, (n, widths[0])), rng.normal(0, 1, (n, widths[-1]))
    lr, wd = 1e-3, 1e-2
    curve = net.train(x, t, epochs=1, batch=batch, lr=lr, weight_decay=wd, seed=1)
    loss_ref, g_ref = ref.loss_and_grad(rounded(p, widths), widths, bf16(x), t)
    assert curve[0] == pytest.approx(loss_ref, rel=2e-2)
    big = np.abs(g_ref) > 0.2 * np.sqrt(np.mean(g_ref ** 2))
    want = p - lr * (np.sign(g_ref) + wd * p)
    # eps = 1e-8 against |g| and FP32 rounding of p: far below 1e-3 of a step
    assert np.abs(net.get_params() - want)[big].max() <= 1e-2 * lr
    net.close()
