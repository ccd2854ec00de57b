"""The sum-factorised FP64 kernels against the generic kernels of the library
(generic_kernels = 1) on the same state: every degree and scheme they cover, boxes
whose cell counts leave ragged 32-cell blocks, axes of one cell, and the three
forms of the stage combination. Both paths are FP64 evaluations of the same
operator in another order: differences are a few hundred roundings of the flux
terms, below 1e-12 of the largest residual."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [("glm", 1), ("glm", 2), ("glm", 3), ("powell", 1), ("powell", 2)]
BOXES = [(1, 1, 1), (3, 1, 2), (5, 4, 3), (33, 2, 1), (8, 9, 4)]


def _state(sol, seed):
    """A smooth positive mean state with modal perturbations (jumps at every face)."""
    import torch
    r = np.random.default_rng(seed)
    w = 0.02 * r.standard_normal((sol.nrows, sol.stride))
    mean = [1.2, 0.3, -0.2, 0.4, 3.0, 0.5, -0.4, 0.3, 0.1]
    rows = sol.mean_rows()
    for k, row in enumerate(rows):
        w[row] = mean[k] * (1.0 + 0.1 * r.standard_normal(sol.stride))
    return torch.as_tensor(w, device="cuda")


@pytest.mark.parametrize("divb,degree", CASES)
@pytest.mark.parametrize("n", BOXES)
def test_matches_generic_kernels(divb, degree, n):
    import torch
    from paper_1806_02343_gb300.binding import Solver
    outs = []
    for generic in (0, 1):
        sol = Solver(3, n, degree, divb, generic_kernels=generic, box_len=0.7)
        w, u0 = _state(sol, 3), _state(sol, 4)
        if divb == "glm":
            sol.set_glm(2.5, 1.7)
        rhs, st0 = torch.zeros_like(w), torch.zeros_like(w)
        sol.rhs(w, None, rhs)
        sol.set_dt(torch.full((1,), 1e-3, dtype=torch.float64, device="cuda"))
        sol.stage(w, None, None, None, st0, None, 0.0, 1.0)
        sol.stage(w, None, u0, None, u0, None, 0.75, 0.25)  # in place on u0
        assert sol.status() == 0
        c = sol.ncell
        outs.append([x[:, :c].cpu().numpy() for x in (rhs, st0, u0)])
    for a, b in zip(*outs):
        assert np.all(np.isfinite(a))
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
