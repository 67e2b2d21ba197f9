"""The order of the network's launches: convolutions that start early (their weights load
while the kernel before them runs) must see the weights and inputs written before them.

Training steps large enough to move every weight, each followed at once by forward passes
and gradients, equal the same passes of a network that was given those weights and waited;
also for inputs that the vector conversion does not take (4 bytes off)."""
import numpy as np
import pytest

from test_gpu_nn import make

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape", [(2, 8, 16), (4, 32, 48), (8, 64, 64), (16, 64, 64), (6, 20, 22)],
                         ids=lambda s: "x".join(map(str, s)))
def test_passes_right_after_an_update(shape):
    from paper_2210_15668_gb300 import ferrox
    net, x, params = make(2, *shape)
    ref, _, _ = make(2, *shape)
    n = int(np.prod(shape))
    xt = torch.as_tensor(x.reshape(-1, 16), dtype=torch.float32, device="cuda")
    off = torch.empty(n * 16 + 1, dtype=torch.float32, device="cuda")[1:].view(n, 16)
    off.copy_(xt)
    tt = torch.as_tensor(np.random.default_rng(4).standard_normal(n), dtype=torch.float32, device="cuda")
    for step in range(6):
        net.loss_grad(xt, tt)
        net.adam_step(1e-2)
        y = net.forward(xt).clone()
        y_off = net.forward(off).clone()
        loss = net.loss_grad(xt, tt)
        torch.cuda.synchronize()
        w, b, gw, gb = net.params()
        ref.set_params(w, b)
        torch.cuda.synchronize()
        y_ref = ref.forward(xt).clone()
        torch.cuda.synchronize()
        assert torch.equal(y, y_ref) and torch.equal(y_off, y_ref), step
        loss_ref = ref.loss_grad(xt, tt)
        _, _, rw, rb = ref.params()
        assert all(np.array_equal(p, q) for p, q in zip(gw + gb, rw + rb)), step
        assert abs(loss - loss_ref) <= 1e-5 * abs(loss_ref)   # its blocks add with atomics
        net.adam_step(1e-30)   # clears the gradients
        ref.adam_step(1e-30)
    net.close()
    ref.close()
