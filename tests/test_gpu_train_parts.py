"""Gradients of more samples than the training kernels' scratch holds at once (2^18):
the sums go on from part to part. The gradient is bit for bit the loop over all
samples, and the first Adam step over such a batch is that gradient's."""
import numpy as np
import pytest

from oracle import mlp as M
from test_gpu_train_order import test_gradient_is_the_loop_over_samples as check_loop

pytestmark = pytest.mark.gpu
PART = 1 << 18


@pytest.mark.parametrize("n", [PART, PART + 1, PART + 300, 2 * PART + 7])
def test_gradient_goes_on_over_the_parts(n):
    check_loop(n, 5)


def test_a_step_over_parts():
    import torch
    from paper_1806_02343_gb300.binding import mlp_loss_grad, mlp_train
    n, nin, lr = PART + 5000, 20, 1e-3
    r = np.random.default_rng(3)
    X = torch.as_tensor(r.normal(size=(n, nin)).astype(np.float32), device="cuda")
    y = (X[:, 0] > 0.5).to(torch.uint8)
    y[: PART // 2] = 1 - y[: PART // 2]
    th = torch.as_tensor(M.init_params(nin, seed=2), dtype=torch.float32, device="cuda")
    want_loss, g = mlp_loss_grad(X, y, th, nin)
    new = th.clone()
    loss = mlp_train(X, y, new, nin, epochs=1, batch=n, lr=lr, seed=5)
    # m = g / 10 and v = g^2 / 1000, both corrected by the same factors: a step of lr g / (|g| + eps)
    big = g.abs() > 1e-3 * g.abs().max()
    step = (new - th)[big].double()
    want = -lr * g[big].double() / (g[big].double().abs() + 1e-8)
    assert big.sum() > 100 and float((step - want).abs().max()) < 1e-3 * lr
    assert abs(loss - want_loss) < 1e-9 * abs(want_loss)
