"""A step size that is positive but rounds to zero in FP32 is a step like any other: it leaves
the weights, moves the moments and clears the gradients.  Adam's second step from a cleared
gradient then moves each weight by lr (b1 m1 / c1) / (sqrt(b2 v1 / c2) + eps) with m1 = (1 - b1) g,
v1 = (1 - b2) g^2: for |g| >> eps by lr (0.09 / 0.19) / sqrt(0.999 / 1.999) = 0.67 lr, to a few FP32
roundings of the weight."""
import numpy as np
import pytest

from test_gpu_nn import make

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tiny", [1e-60, 5e-324])
def test_step_size_below_fp32_is_a_step(tiny):
    net, x, _ = make(4, 4, 8, 16)
    t = np.random.default_rng(5).standard_normal(4 * 8 * 16)
    net.loss_grad(torch.as_tensor(x.reshape(-1, 16), dtype=torch.float32, device="cuda"),
                  torch.as_tensor(t, dtype=torch.float32, device="cuda"))
    w0, b0, gw, gb = net.params()
    net.adam_step(tiny)
    w1, b1, gw1, gb1 = net.params()
    lr = 1e-3
    net.adam_step(lr)
    w2, b2, _, _ = net.params()
    net.close()
    assert max(np.abs(g).max() for g in gw + gb) > 1e-2
    for a, b in zip(w0 + b0, w1 + b1):
        assert np.array_equal(a, b)
    assert all(not np.any(g) for g in gw1 + gb1)
    move = lr * (0.09 / 0.19) / np.sqrt(0.999 / 1.999)
    for a, b, g in zip(w0 + b0, w2 + b2, gw + gb):
        big = np.abs(g) > 1e-4   # eps is 1e-4 of it
        assert np.abs((a - b)[big] - np.sign(g[big]) * move).max(initial=0.0) <= 1e-3 * move + 2e-7 * np.abs(a).max()
