"""The step network's gradient and optimiser step at the sizes where the
training kernel's tiles can go wrong: fewer samples than a tile, whole tiles,
remainders, and more tiles than blocks."""
import numpy as np
import pytest
import torch

import oracle.stepnet as OS

pytestmark = pytest.mark.gpu


def _data(n):
    g = np.random.Generator(np.random.Philox(77 + n))
    x = g.normal(0.0, 1.0, (n, 8)).astype(np.float32)
    return x, (6.0 + g.normal(0.0, 1.0, n)).astype(np.float32)


@pytest.mark.parametrize("n", [1, 15, 31, 32, 33, 4096, 9728, 20011])
def test_gradient_against_fp64(n):
    from paper_1901_10475_gb300.stepnet import StepNet
    torch.cuda.set_device(0)
    x, t = _data(n)
    net = StepNet(seed=5)
    dx, dt = torch.as_tensor(x, device="cuda"), torch.as_tensor(t, device="cuda")
    loss, grad = net.grad(dx, dt)
    want_loss, want = OS.loss_and_grad(net.params, x, t)
    # FP32 sums of products against FP64: 1e-3 of the largest component, as
    # for the other gradient checks
    assert abs(loss - want_loss) <= 1e-5 * abs(want_loss)
    assert np.abs(grad.cpu().numpy() - want).max() <= 1e-3 * np.abs(want).max()
    # summed in a fixed order: the same bits again
    loss2, grad2 = net.grad(dx, dt)
    assert loss2 == loss and torch.equal(grad2, grad)
    # one AdamW step from that gradient: m = 0.1 g, v = 0.001 g^2, both
    # corrected to g and g^2, then decoupled decay of the weights
    p0, g, lr, wd = net.params.astype(np.float64), grad.cpu().numpy().astype(np.float64), 1e-3, 0.1
    assert net.train_step(dx, dt, lr, wd) == loss
    weight = np.ones(4801, bool)
    weight[512:576] = weight[4672:4736] = weight[4800:] = False
    ref = p0 * np.where(weight, 1.0 - lr * wd, 1.0) - lr * g / (np.abs(g) + 1e-8)
    assert np.abs(net.params - ref).max() <= 1e-6 + 1e-4 * lr
    net.close()
