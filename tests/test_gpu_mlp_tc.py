"""The two forms of the fused tensor-core inference (one 128-row tile per SM at most: deep ring of weight copies; more: two
CTAs per SM, shallow ring) over widths that divide neither the copies' 32 columns nor the swizzled blocks of 64, layers
narrower than 16 and the widest, several copies per slot and several slots per layer. Against the CPU oracle on BF16
weights and inputs, within the bounds of the other serving tests: 2e-2 of the largest output (BF16 activations); and a
row's outputs do not depend on how many rows there are (the same arithmetic in the same order): bitwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def bf16(a):
    u = np.ascontiguousarray(a, dtype=np.float32).view(np.uint32)
    return (((u + 0x7FFF + ((u >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32).astype(np.float64)


def bf16_weights(p, widths):
    q = np.array(p, dtype=np.float64)
    off = 0
    for a, b in zip(widths[:-1], widths[1:]):
        q[off:off + a * b] = bf16(q[off:off + a * b])
        off += a * b + b
    return q


@pytest.mark.parametrize("widths", [[6, 256, 256, 256, 4], [5, 40, 72, 200, 9], [20, 256, 16, 33, 130, 3],
                                    [3, 1, 5], [256, 256], [100, 17, 250, 241]])
def test_tensor_core_forms(widths):
    import torch
    from oracle import mlp as ref
    from paper_1009_2727_gb300.surrogate import MLP
    rng = np.random.default_rng(23)
    net = MLP(widths, seed=4)
    p = net.get_params().astype(np.float64)
    net.set_params(p + rng.normal(0, 0.05, p.size))
    pq = bf16_weights(net.get_params(), widths)
    tiles = torch.cuda.get_device_properties(0).multi_processor_count
    x = rng.normal(0, 1, (128 * tiles + 77, widths[0]))
    many = net.forward(x)
    for n in (1, 129, 128 * tiles):
        few = net.forward(x[:n])
        assert np.array_equal(few, many[:n]), n
    rows = np.r_[0:200, len(x) - 200:len(x)]
    y_ref, _ = ref.forward(pq, widths, bf16(x[rows]))
    assert np.abs(many[rows] - y_ref).max() <= 2e-2 * np.abs(y_ref).max()
    net.close()
