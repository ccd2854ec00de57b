"""The tiled inference kernel (FP32 form, x-rows of whole 128-cell tiles) over its
degrees and schemes, on meshes whose tiles wrap onto themselves (one tile per row,
axes of one cell) and on two tiles per row: probabilities against the FP64 network
on the oracle's features, to the 0.03 that BF16 features and weights allow, and the
flags where the probability is not that close to the threshold."""
import numpy as np
import pytest

from oracle import mlp as M
from oracle.dg import Scheme
from gpu_helpers import means_to_device, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("d", [1, 2, 3])
@pytest.mark.parametrize("n", [(128, 1, 1), (128, 3, 2), (256, 2, 3)])
def test_probabilities_match_the_fp64_network(divb, d, n):
    import torch
    from paper_1806_02343_gb300.binding import DG_LIMIT_MLP, DG_PREC_FP32MIX, Solver
    S = Scheme(3, d, divb, 5.0 / 3.0, n)
    r = np.random.default_rng(11)
    w0 = 0.05 * r.normal(size=(S.C, S.N)) * np.exp(r.normal(size=(S.C, 1)))
    mean = [1.0, 0.4, -0.3, 0.2, 3.0, 0.6, -0.5, 0.4, 0.1]
    for k, row in enumerate(np.flatnonzero(S.is_mean)):
        w0[:, row] = mean[k] * (1.0 + 0.2 * r.normal(size=S.C))
    w0 = w0.astype(np.float32).astype(np.float64)
    sol = Solver(3, n, d, divb, gamma=5.0 / 3.0, box_len=S.L, precision=DG_PREC_FP32MIX, limiter=DG_LIMIT_MLP)
    th = M.init_params(sol.n_features(), seed=5)
    X = M.features(S, w0)
    z, _ = M.forward(th, X)
    th[-1] -= float(np.median(z))
    z, _ = M.forward(th, X)
    p_ref = M.sigmoid(z)
    sol.mlp_set_weights(torch.as_tensor(th, dtype=torch.float32, device="cuda"), 0.5)
    flags = torch.zeros(sol.stride, dtype=torch.uint8, device="cuda")
    prob = torch.zeros(sol.stride, dtype=torch.float32, device="cuda")
    sol.mlp_infer(to_device(w0, sol), means_to_device(w0, sol, S), flags, prob)
    assert sol.status() == 0
    p = prob[: sol.ncell].cpu().numpy()
    assert np.max(np.abs(p - p_ref)) < 0.03
    sure = np.abs(p_ref - 0.5) > 0.03
    assert sure.any() and np.array_equal(flags[: sol.ncell].cpu().numpy()[sure].astype(bool), (p_ref > 0.5)[sure])
