"""Positivity of FP64 states: the FP32 pre-screen and the list kernel. Cells whose
pressure dips at one of the scheme's points each, below the floor or just above
it; cells whose density does; cells whose mean pressure or density is below its
floor; one with a coefficient that is not a number (comparisons fail, so it stays).
Limited cells agree with the oracle to 1e-12 (some hundred roundings, and the
factor's division by a pressure difference of order one), the others bit for bit."""
import numpy as np
import pytest

from oracle.dg import Scheme
from oracle.limiter import Limiter
from paper_1806_02343_gb300 import workloads as W
from gpu_helpers import from_device, rel_err, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("copies", [1, 60])
def test_fp64_cells_are_limited_as_the_oracle(divb, d, copies):
    from paper_1806_02343_gb300.binding import Solver
    npt = (d + 1) ** 3 + 6 * (d + 1) ** 2
    n = (npt, 4, copies)
    S = Scheme(3, d, divb, 5.0 / 3.0, (npt, 4, 1))
    w0 = S.project(lambda x: W.uniform_state(x, nvar=S.V, rho=1.0, v=(2.0, 1.0, -1.0), p=1.0, B=(0.3, 0.2, 0.1)))
    gm1 = S.gamma - 1.0
    for var, half, low in ((4, 0, -0.02), (4, 1, 0.05), (0, 2, -0.1)):  # lowest pressure, or density, over the points
        rows = slice(var * S.n, (var + 1) * S.n)
        P = np.concatenate([S.Sv[rows, :, var]] + [S.Sf[a, s][rows, :, var] for a in range(3) for s in (-1, 1)], 1)
        K = np.einsum("lp,l,lq->pq", P[1:], 1.0 / S.mass[rows][1:], P[1:])  # [point, centre]
        amp = (1.0 - low) / (gm1 if var == 4 else 1.0) / K.max(0)
        w0[half * npt:(half + 1) * npt, var * S.n + 1:(var + 1) * S.n] -= (amp[:, None] * P[1:].T) / S.mass[rows][1:]
    w0[3 * npt, 4 * S.n] = 2.0       # mean pressure below the floor
    w0[3 * npt + 1, 0] = -0.5        # mean density below the floor
    ref = Limiter(S, tvb=False, positivity=True).positivity(w0)
    w0[3 * npt + 2, 2] = ref[3 * npt + 2, 2] = np.nan
    changed = np.any((ref != w0) & ~np.isnan(ref), 1)
    assert changed[:npt].all() and not changed[npt:2 * npt].any() and changed[2 * npt:3 * npt + 2].all()
    sol = Solver(3, n, d, divb, positivity=1)
    S.C, many, refs = sol.ncell, np.tile(w0, (copies, 1)), np.tile(ref, (copies, 1))
    w = to_device(many, sol)
    sol.limit(w, None)
    got = from_device(w, sol)
    same = np.tile(~changed, copies)
    assert np.array_equal(got[same], many[same], equal_nan=True)
    # (a mean set to the floor exactly makes the oracle's factor 0 / 0: its rows beyond the means are left out)
    fin = np.isfinite(refs) & ~same[:, None]
    assert np.all(np.isfinite(got[~same])) and fin[:, S.is_mean][~same].all()
    assert rel_err(got[fin], refs[fin]) < 1e-12
