"""The smoothness indicator from the non-zero entries of its forms: every degree,
scheme and dimension on a state whose coefficients are all non-zero, against the
oracle's dense forms (1e-11 of the largest value, as in the regridding tests)."""
import numpy as np
import pytest

from oracle import regrid as G
from oracle.dg import Scheme
from gpu_helpers import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("dim,degree", [(2, 1), (2, 2), (2, 3), (3, 1), (3, 2), (3, 3)])
@pytest.mark.parametrize("fields", [(0,), (5, 6, 7), (0, 1, 2, 3, 4, 5, 6, 7)])
def test_every_form(divb, dim, degree, fields):
    from paper_1806_02343_gb300.binding import Solver
    n = (7, 5, 4)[:dim]
    S = Scheme(dim, degree, divb, 5.0 / 3.0, n)
    w0 = np.random.default_rng(4).normal(size=(S.C, S.N))
    ref = G.smoothness(S, w0, fields).reshape(S.C, -1).max(axis=1)
    sol = Solver(dim, n, degree, divb, gamma=5.0 / 3.0, box_len=S.L)
    got = sol.smoothness(to_device(w0, sol), None, fields).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-11 * ref.max()
