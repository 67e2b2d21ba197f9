"""Weight and bias gradients on grids that leave ragged 16 x 8 x tz tiles, wrap the halo
around sides shorter than it, and give several tiles to a block, against the oracle's
layers with BF16 storage emulated (the bound of test_gpu_nn: 2e-2 normwise), and the same
bits on a second run (the blocks' sums are added in a fixed order)."""
import numpy as np
import pytest

from test_gpu_nn import forward_backward_bf16_storage, make, rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape", [(2, 2, 2), (2, 10, 18), (6, 4, 34), (4, 48, 32), (10, 18, 6), (12, 64, 128)],
                         ids=lambda s: "x".join(map(str, s)))
def test_gradients_on_ragged_grids(shape):
    net, x, params = make(2, *shape)
    t = np.random.default_rng(3).standard_normal(shape)
    xt = torch.as_tensor(x.reshape(-1, 16), dtype=torch.float32, device="cuda")
    tt = torch.as_tensor(t.ravel(), dtype=torch.float32, device="cuda")
    loss = net.loss_grad(xt, tt)
    _, _, gw, gb = net.params()
    net.adam_step(1e-12)   # clears the gradients
    net.loss_grad(xt, tt)
    _, _, gw2, gb2 = net.params()
    net.close()
    assert all(np.array_equal(a, b) for a, b in zip(gw + gb, gw2 + gb2))
    loss_or, g_or = forward_backward_bf16_storage(params, x, t)
    assert abs(loss - loss_or) <= 2e-2 * loss_or
    for layer in range(6):
        e_w = rel(gw[layer], g_or[layer][0].reshape(27, *g_or[layer][0].shape[3:]))
        e_b = rel(gb[layer], g_or[layer][1])
        assert e_w <= 2e-2 and e_b <= 2e-2, (layer, e_w, e_b)
