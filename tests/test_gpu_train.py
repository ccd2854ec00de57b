"""Loss and gradient of the indicator's training kernels against the FP64 oracle
at the edges of their tiles: 32-sample tiles (one sample, a ragged last tile, more
tiles than blocks), 128-input passes (one input, a ragged pass, several passes).
Tolerances as in test_gpu_mlp.py: FP32 sums of up to 1e4 terms."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nin", [(1, 110), (31, 1), (33, 62), (257, 128), (500, 129), (300, 300), (10000, 110)])
def test_loss_and_gradient(n, nin):
    import torch
    from paper_1806_02343_gb300.binding import mlp_loss_grad
    rng = np.random.default_rng(n + nin)
    X = rng.normal(size=(n, nin)).astype(np.float32)
    y = (X.sum(1) > 0.3).astype(np.uint8)
    th = M.init_params(nin, seed=4).astype(np.float32)
    th[M.H * nin:M.H * nin + M.H] = rng.normal(0, 0.1, M.H)
    ref_loss, ref = M.loss_and_grad(th.astype(np.float64), X.astype(np.float64), y.astype(float), pos_weight=3.0)
    loss, g = mlp_loss_grad(torch.as_tensor(X, device="cuda"), torch.as_tensor(y, device="cuda"),
                            torch.as_tensor(th, device="cuda"), nin, pos_weight=3.0)
    assert abs(loss - ref_loss) < 1e-5 * abs(ref_loss)
    assert np.max(np.abs(g.cpu().numpy() - ref)) < 1e-4 * np.max(np.abs(ref))


def test_steps_repeat_bitwise():
    """The gradient's sums run in a fixed order: two trainings from one seed agree bit for bit."""
    import torch
    from paper_1806_02343_gb300.binding import mlp_train
    rng = np.random.default_rng(1)
    X = torch.as_tensor(rng.normal(size=(3000, 112)).astype(np.float32), device="cuda")
    y = (X[:, 0] > 0.5).to(torch.uint8)
    out = []
    for _ in range(2):
        th = torch.as_tensor(M.init_params(110, seed=2), dtype=torch.float32, device="cuda")
        mlp_train(X, y, th, 110, epochs=2, batch=700, lr=1e-3, seed=5)
        out.append(th)
    assert torch.equal(*out)
