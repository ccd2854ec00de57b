"""The positivity limiter does not depend on the units of the state: densities,
momenta, energies and floors multiplied by a power of four (fields by its square
root, so velocities stay) give the result multiplied by it, bit for bit, since
every operation of the procedure scales exactly. States planted with cells whose
pressure or density dips below the floor at one point each, and with means below
it; the FP32 form where its rows stay ordinary FP32 numbers although products of
two of them do not, FP64 also far outside the range of FP32."""
import numpy as np
import pytest

from oracle.dg import Scheme
from oracle.limiter import Limiter
from paper_1806_02343_gb300 import workloads as W
from gpu_helpers import from_device, means_to_device, to_device

pytestmark = pytest.mark.gpu


def _planted(d, divb):
    npt = (d + 1) ** 3 + 6 * (d + 1) ** 2
    S = Scheme(3, d, divb, 5.0 / 3.0, (npt, 4, 1))
    w = S.project(lambda x: W.uniform_state(x, nvar=S.V, rho=1.0, v=(2.0, 1.0, -1.0), p=1.0, B=(0.3, 0.2, 0.1)))
    for var, part, low in ((4, 0, -0.02), (4, 1, 0.05), (0, 2, -0.1)):
        rows = slice(var * S.n, (var + 1) * S.n)
        P = np.concatenate([S.Sv[rows, :, var]] + [S.Sf[a, s][rows, :, var] for a in range(3) for s in (-1, 1)], 1)
        K = np.einsum("lp,l,lq->pq", P[1:], 1.0 / S.mass[rows][1:], P[1:])
        amp = (1.0 - low) / (S.gamma - 1.0 if var == 4 else 1.0) / K.max(0)
        w[part * npt:(part + 1) * npt, var * S.n + 1:(var + 1) * S.n] -= (amp[:, None] * P[1:].T) / S.mass[rows][1:]
    w[3 * npt, 4 * S.n] = 2.0   # mean pressure below the floor
    w[3 * npt + 1, 0] = -0.5    # mean density below the floor
    w = w.astype(np.float32).astype(np.float64)
    w[np.abs(w) < 1e-12] = 0.0  # the projection's rounding, which the smaller units would push out of FP32
    hit = np.any(Limiter(S, tvb=False, positivity=True).positivity(w) != w, 1)
    assert hit[:npt].all() and not hit[npt:2 * npt].any() and hit[2 * npt:3 * npt + 2].all()
    return S, w, hit


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("prec,e", [("fp64", -40), ("fp64", -100), ("fp64", 100), ("fp32", -40), ("fp32", 25)])
def test_limited_state_scales(divb, d, prec, e):
    from paper_1806_02343_gb300.binding import DG_PREC_FP32MIX, DG_PREC_FP64, Solver
    S, w0, hit = _planted(d, divb)
    field = np.any(S.Sv[:, :, 5:8] != 0.0, (1, 2))
    outs = []
    for k in (0, e):
        f = np.where(field, 2.0 ** k, 4.0 ** k)
        sol = Solver(3, S.ncell, d, divb, positivity=1,
                     precision=DG_PREC_FP32MIX if prec == "fp32" else DG_PREC_FP64,
                     eps_rho=1e-6 * 4.0 ** k, eps_p=1e-6 * 4.0 ** k)
        w = to_device(w0 * f, sol)
        wm = means_to_device(w0 * f, sol, S) if sol.fp32 else None
        sol.limit(w, wm)
        outs.append(from_device(w, sol) / f)
        assert np.array_equal(np.any(outs[-1] != w0, 1), hit)
    assert np.array_equal(*outs)
