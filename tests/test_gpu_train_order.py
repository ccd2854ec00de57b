"""Weight gradients of the training kernels are sums over the samples in their
order, products and sums rounded separately in FP32, for each layer and the biases:
bit for bit a loop on the host, on weights that make every other sum exact (hidden
activations 1, output 0). Sample counts at the edges of the 256-sample chunks."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.mark.parametrize("n,nin", [(1, 3), (255, 110), (256, 16), (3001, 110)])
def test_gradient_is_the_loop_over_samples(n, nin):
    import torch
    from paper_1806_02343_gb300.binding import mlp_loss_grad
    r = np.random.default_rng(n)
    X = r.normal(size=(n, nin)).astype(F)
    y = (r.random(n) < 0.3).astype(np.uint8)
    H = M.H
    th = np.concatenate([np.zeros(H * nin), np.ones(H),              # h1 = 1
                         np.full(H * H, 2.0 ** -6), np.zeros(H),     # h2 = 64 / 64
                         np.ones(H), [-64.0]]).astype(F)             # z = 0, p = 1 / 2
    _, g = mlp_loss_grad(torch.as_tensor(X, device="cuda"), torch.as_tensor(y, device="cuda"),
                         torch.as_tensor(th, device="cuda"), nin, pos_weight=3.0)
    d3 = np.where(y, F(-1.5), F(0.5)) * F(1.0 / F(n))
    d1 = np.zeros(n, F)
    for _ in range(H):
        d1 = d1 + d3 * F(2.0 ** -6)  # the product is exact
    s3, s1, w1 = F(0), F(0), np.zeros(nin, F)
    for b in range(n):
        s3 = s3 + d3[b]
        s1 = s1 + d1[b]
        w1 = w1 + d1[b] * X[b]
    want = np.concatenate([np.tile(w1, H), np.full(H, s1), np.full(H * H, s3), np.full(H, s3), np.full(H, s3), [s3]])
    assert want.dtype == F and np.array_equal(g.cpu().numpy(), want)
