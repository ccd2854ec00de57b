"""Point-wise positivity screen of the FP32 form: cells whose pressure dips at one
of the scheme's volume or face points each, below the floor in one half of the
cells and just above it in the other. Exactly the first half is limited (as in the
oracle), the second half comes back bit for bit. Short lists put one cell on a
warp, longer ones up to 32: both kinds."""
import numpy as np
import pytest

from oracle.dg import Scheme
from oracle.limiter import Limiter
from paper_1806_02343_gb300 import workloads as W
from gpu_helpers import from_device, means_to_device, rel_err, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("copies", [1, 400])
def test_each_point_is_seen(divb, d, copies):
    from paper_1806_02343_gb300.binding import DG_PREC_FP32MIX, Solver
    npt = (d + 1) ** 3 + 6 * (d + 1) ** 2
    n = (npt, 2, copies)
    S = Scheme(3, d, divb, 5.0 / 3.0, (npt, 2, 1))
    w0 = S.project(lambda x: W.uniform_state(x, nvar=S.V, rho=1.0, v=(2.0, 1.0, -1.0), p=1.0, B=(0.3, 0.2, 0.1)))
    rows = slice(4 * S.n, 5 * S.n)
    P = np.concatenate([S.Sv[rows, :, 4]] + [S.Sf[a, s][rows, :, 4] for a in range(3) for s in (-1, 1)], 1)
    K = np.einsum("lp,l,lq->pq", P[1:], 1.0 / S.mass[rows][1:], P[1:])     # [point, centre]
    gm1 = S.gamma - 1.0
    for half, p_low in ((0, -0.02), (1, 0.05)):
        amp = (1.0 - p_low) / gm1 / K.max(0)                              # lowest pressure over the points: p_low
        w0[half * npt:(half + 1) * npt, 4 * S.n + 1:5 * S.n] -= (amp[:, None] * P[1:].T) / S.mass[rows][1:]
    w0 = w0.astype(np.float32).astype(np.float64)
    ref = Limiter(S, tvb=False, positivity=True).positivity(w0)
    assert np.array_equal(np.any(ref != w0, 1), np.arange(2 * npt) < npt)
    sol = Solver(3, n, d, divb, precision=DG_PREC_FP32MIX, positivity=1)
    S.C, many, refs = sol.ncell, np.tile(w0, (copies, 1)), np.tile(ref, (copies, 1))
    w, wm = to_device(many, sol), means_to_device(many, sol, S)
    sol.counters(reset=True)
    sol.limit(w, wm)
    got = from_device(w, sol)
    assert sol.counters()["pos_cells"] == npt * copies
    same = np.tile(np.arange(2 * npt) >= npt, copies)
    assert np.array_equal(got[same], many[same])
    assert rel_err(got, refs) < 1e-5
