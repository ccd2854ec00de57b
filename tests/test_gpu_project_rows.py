"""FP64 projection: the kernel with lanes over cells forms every row's sum in the
order and rounding of the generic one (rows of the state, bit for bit), for each
degree, scheme and number of points, on a box with a ragged 128-cell block."""
import pytest
import torch

from oracle.dg import Scheme
from gpu_helpers import nodal_input, nodal_to_device
from test_gpu_project import _field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("degree,npts", [(1, 1), (1, 2), (1, 3), (2, 3), (2, 4), (2, 6), (3, 3), (3, 4), (3, 5)])
def test_fp64_rows_equal_the_generic_ones(divb, degree, npts):
    from paper_1806_02343_gb300.binding import Solver
    n = (7, 5, 4)
    S = Scheme(3, degree, divb, 5.0 / 3.0, n)
    out = []
    for generic in (0, 1):
        sol = Solver(3, n, degree, divb, generic_kernels=generic)
        w, _ = sol.alloc_state()
        sol.project(nodal_to_device(nodal_input(S, lambda x: _field(x, S.V), npts), sol), npts, w, None)
        out.append(w[:, : sol.ncell].clone())
    assert torch.equal(out[0], out[1])
