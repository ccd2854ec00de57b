"""The projection kernels against the oracle's L2 projection with the same number
of points: every (degree, points) pair of the sum-factorised kernel and, beyond
its range, the dense one; a box that leaves a ragged 32-cell block. FP64 sums of
at most 216 products: 1e-13 of the largest coefficient; FP32 rows one rounding."""
import numpy as np
import pytest

from oracle.dg import Scheme
from gpu_helpers import from_device, mean_rows, nodal_input, nodal_to_device

pytestmark = pytest.mark.gpu

PAIRS = [(1, 1), (1, 2), (1, 3), (1, 4), (2, 3), (2, 4), (2, 5), (2, 6), (3, 3), (3, 4), (3, 5), (3, 6)]


def _field(x, V):
    u = np.stack([np.cos((1 + 0.3 * v) * x[..., 0] + 2 * x[..., 1] - x[..., 2] + v) for v in range(V)], -1)
    u[..., 0] += 3.0
    return u


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("degree,npts", PAIRS)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_projection_matches_oracle(divb, degree, npts, prec):
    from paper_1806_02343_gb300.binding import DG_PREC_FP32MIX, DG_PREC_FP64, Solver
    n = (5, 4, 2)
    S = Scheme(3, degree, divb, 5.0 / 3.0, n)
    fn = lambda x: _field(x, S.V)  # noqa: E731
    sol = Solver(3, n, degree, divb, precision=DG_PREC_FP32MIX if prec == "fp32" else DG_PREC_FP64)
    w, wm = sol.alloc_state()
    sol.project(nodal_to_device(nodal_input(S, fn, npts), sol), npts, w, wm)
    ref = S.project(fn, npts)
    top = np.max(np.abs(ref))
    err = np.max(np.abs(from_device(w, sol) - ref))
    assert err <= (1e-13 if prec == "fp64" else 6e-8) * top
    if prec == "fp32":
        assert np.max(np.abs(wm[:, : sol.ncell].cpu().numpy().T - ref[:, mean_rows(S)])) <= 1e-13 * top
