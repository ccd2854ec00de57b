"""The FP64 kernels of uniform 2D meshes against the generic kernels of the library
(generic_kernels = 1) on the same state: every degree and scheme, meshes that leave
ragged blocks (32 cells of a face block, 4 of a cell block), axes of one cell, the
three forms of the stage combination, and the timestep with its scalars, twice.
Both paths are FP64 evaluations of the same operator in another order: differences
are a few hundred roundings of the flux terms, below 1e-12 of the largest residual;
the timestep is some dozen operations: 1e-13."""
import numpy as np
import pytest

from test_gpu_sf import _state

pytestmark = pytest.mark.gpu

MESHES = [(1, 1), (1, 3), (5, 7), (33, 2), (24, 24), (300, 280)]


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("n", MESHES)
def test_matches_generic_kernels(divb, degree, n):
    import torch
    from paper_1806_02343_gb300.binding import Solver
    outs, dts = [], []
    for generic in (0, 1):
        sol = Solver(2, n, degree, divb, generic_kernels=generic, box_len=0.7)
        w, u0 = _state(sol, 3), _state(sol, 4)
        if divb == "glm":
            sol.set_glm(2.5, 1.7)
        rhs, st0 = torch.zeros_like(w), torch.zeros_like(w)
        sol.rhs(w, None, rhs)
        sol.set_dt(torch.full((1,), 1e-3, dtype=torch.float64, device="cuda"))
        sol.stage(w, None, None, None, st0, None, 0.0, 1.0)
        sol.stage(w, None, u0, None, u0, None, 0.75, 0.25)  # in place on u0
        dt = torch.zeros(2, dtype=torch.float64, device="cuda")
        sol.dt(w, None, dt[0:])
        sol.dt(u0, None, dt[1:])
        assert sol.status() == 0
        speeds = sol.glm_speeds() if divb == "glm" else (0.0, 0.0)
        c = sol.ncell
        outs.append([x[:, :c].cpu().numpy() for x in (rhs, st0, u0)])
        dts.append(np.array([*dt.cpu().numpy(), *speeds]))
    for a, b in zip(*outs):
        assert np.all(np.isfinite(a))
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
    assert np.all(np.abs(dts[0] - dts[1]) <= 1e-13 * np.abs(dts[1]))
