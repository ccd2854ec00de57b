"""The TVB limiter of FP64 states does not depend on their units: with no threshold
(Mtilde = 0, tvb_eps = 0), densities, momenta and energies multiplied by a power of
four, fields (and psi) by its square root, give the result multiplied by it, bit for
bit: every operation of the procedure scales exactly, and the cells it runs on must
include all that it changes. A ramp of the density along x in a gas at rest (an
entropy wave), slopes 1e-3 below their limit in one half of the cells (kept) and
1e-3 above it in the other (limited); units inside FP32's range, at its ends and far
outside."""
import numpy as np
import pytest

from oracle import mhd
from oracle.dg import Scheme
from gpu_helpers import from_device, to_device
from test_gpu_tvb_margins import G, _fill

pytestmark = pytest.mark.gpu
N = (16, 9, 8)


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("rise", [1e-2, 1e-5])
@pytest.mark.parametrize("k", [-10, -40, -50, -55, -58, -60, -62, -64, -70, -100, 40, 55, 60, 64, 100])
def test_limited_state_scales(divb, d, rise, k):
    import torch
    from paper_1806_02343_gb300.binding import DG_LIMIT_TVB, Solver
    S = Scheme(3, d, divb, G, N)
    r = np.random.default_rng(2)
    C, i = S.C, np.arange(S.C) % N[0]
    rho = 1.0 + rise * i
    u = mhd.conserved(rho, np.zeros((C, 3)), np.full(C, 0.8), np.tile([0.5, 0.3, -0.7], (C, 1)), G)
    if S.V == 9:
        u = np.concatenate([u, np.full((C, 1), 0.2)], 1)
    sl = np.zeros((C, 3, S.V))
    sl[:, 0, 0] = 0.5 * S.P.beta * rise * (1.0 + 1e-3 * r.choice([-1.0, 1.0], C))
    w0, _ = _fill(S, u, sl)
    if d == 2:
        w0[:, S.modes.index((2, 0, 0))] = 1e-3 * rise
    field = np.any(S.Sv[:, :, 5:] != 0.0, (1, 2))
    outs = []
    for e in (0, k):
        f = np.where(field, 2.0 ** e, 4.0 ** e)
        sol = Solver(3, N, d, divb, gamma=G, box_len=S.L, Mtilde=0.0, tvb_eps=0.0, limiter=DG_LIMIT_TVB)
        if divb == "glm":
            sol.set_glm(3.0, 1.0)
        w = to_device(w0 * f, sol)
        flags = torch.zeros(sol.stride, dtype=torch.uint8, device="cuda")
        sol.limit(w, None, flags)
        outs.append((flags[:C].cpu().numpy(), from_device(w, sol) / f))
    (h0, a), (h1, b) = outs
    assert C // 4 < h0.sum() < 3 * C // 4
    assert np.array_equal(h0, h1) and np.array_equal(a, b)
