"""Margins of the conservative detector in front of the TVB procedure, where its
arithmetic and the procedure's differ most. The listed cells must contain every
cell that the procedure changes, so the changed cells and the state are those of
the procedure on every cell."""
import numpy as np
import pytest

from oracle import mhd
from oracle.dg import Scheme
from oracle.limiter import Limiter
from gpu_helpers import from_device, means_to_device, to_device

pytestmark = pytest.mark.gpu
G = 5.0 / 3.0


def _fill(S, u, slopes):
    """Oracle state of cell means u [C, V] and slopes along the axes [C, 3, V], B without slopes of its own axis."""
    w = np.zeros((S.C, S.N))
    lim = Limiter(S, tvb=True, positivity=False)
    for k in range(9 if S.divb == "glm" else 5):
        w[:, k * S.n] = u[:, k]
        for a in range(3):
            w[:, k * S.n + lim.deg1[a]] = slopes[:, a, k]
    if S.divb == "powell":
        for j in range(len(S.ldf)):
            if lim.ldf_deg[j] <= 1:
                w[:, 5 * S.n + j] = (u[:, 5:8] @ lim.proj_const[j]
                                     + np.einsum("kac,ca->k", slopes[:, :, 5:8], lim.proj_lin[j]))
    return w, lim


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_fp32_near_the_double_degeneracy(d, axis):
    """a = c_A with a vanishing transverse field: the gap c_f^2 - c_s^2 is at rounding level, and the procedure's
    FP32 eigenvector weights exceed 1 by what that rounding makes of them. Transverse-field slopes whose amplitude
    would stay below the threshold with weights of at most 1: cells change only where the weights exceed it."""
    import torch
    from paper_1806_02343_gb300.binding import DG_LIMIT_TVB, DG_PREC_FP32MIX, Solver
    from paper_1806_02343_gb300.workloads import morton_order
    L = 4
    m = 2 ** L
    S = Scheme(3, d, "powell", G, (m, m, m))
    r = np.random.default_rng(11 + axis)
    C, t1 = S.C, (axis + 1) % 3
    rho, p = np.full(C, 1.0), np.full(C, 0.6)
    bn = np.sqrt(G * 0.6) * (1.0 + np.exp(r.uniform(-8.0, -7.0, C)) * r.choice([-1.0, 1.0], C))
    B = np.zeros((C, 3))
    B[:, axis] = bn
    B[:, t1] = bn * np.exp(r.uniform(-13.0, -10.0, C))
    u = mhd.conserved(rho, np.zeros((C, 3)), p, B, G)
    thr = 0.1
    sl = np.zeros((C, 3, 8))
    sl[:, axis, 5 + t1] = thr * r.uniform(0.8, 0.97, C) * 2.0 * np.sqrt(rho * G * p / rho)  # (1/2) db / (sqrt(rho) a)
    w0, _ = _fill(S, u, sl)
    w0 = w0.astype(np.float32).astype(np.float64)
    ijk = np.array([(i, j, k) for k in range(m) for j in range(m) for i in range(m)], dtype=np.int32)
    lev = np.full(C, L, np.int8)
    order = morton_order(lev, ijk, 3, L)
    outs = []
    for perm, kw in ((np.arange(C), {}), (order, dict(levels=lev[order], ijk=ijk[order]))):
        sol = Solver(3, None if kw else (m, m, m), d, "powell", gamma=G, box_len=S.L, Mtilde=thr / S.dx,
                     limiter=DG_LIMIT_TVB, precision=DG_PREC_FP32MIX, **kw)
        w = to_device(w0[perm], sol)
        flags = torch.zeros(sol.stride, dtype=torch.uint8, device="cuda")
        sol.limit(w, means_to_device(w0[perm], sol, S), flags)
        hit, full = np.zeros(C, bool), np.zeros_like(w0)
        hit[perm] = flags[:C].cpu().numpy().astype(bool)
        full[perm] = from_device(w, sol)
        outs.append((hit, full))
    (h0, w_all), (h1, w_list) = outs
    assert 10 < h0.sum() < C // 2
    assert np.array_equal(h0, h1) and np.array_equal(w_all, w_list)


@pytest.mark.parametrize("divb", ["glm", "powell"])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("size", [1e-2, 1e-3, 1e-4, 1e-6])
def test_fp64_small_increments_on_a_background(divb, d, size):
    """Entropy waves of a part `size` of the mean, slopes within 4e-8 / size of the limit that the smaller neighbour
    difference sets: the differences of the means lose their digits if the means are rounded to FP32 first."""
    import torch
    from paper_1806_02343_gb300.binding import DG_LIMIT_TVB, Solver
    n = (12, 9, 8)
    S = Scheme(3, d, divb, G, n)
    S.P.Mtilde = 1e-9 / S.dx
    S.P.tvb_eps = 0.0
    r = np.random.default_rng(3)
    C = S.C
    i = np.arange(C) % n[0]
    x = size * np.cumsum(r.uniform(0.5, 1.5, n[0]))       # rising along x, one step back at the period
    rho = 1.0 + x[i]
    v = np.array([0.7, -0.4, 0.3])
    B = np.array([0.5, 0.3, -0.6])
    u = mhd.conserved(rho, np.tile(v, (C, 1)), np.full(C, 0.8), np.tile(B, (C, 1)), G)
    if S.V == 9:
        u = np.concatenate([u, np.zeros((C, 1))], 1)
    dp, dm = 0.5 * (rho[S.nbr_plus[0]] - rho), 0.5 * (rho - rho[S.nbr_minus[0]])
    s = S.P.beta * np.minimum(dp, dm) * (1.0 + np.minimum(4e-8 / size, 0.3) * r.uniform(-1.0, 1.0, C))
    sl = np.zeros((C, 3, S.V))
    s = np.where((dp > 0) & (dm > 0), s, 0.0)
    sl[:, 0, 0] = s
    sl[:, 0, 1:4] = s[:, None] * v
    sl[:, 0, 4] = s * 0.5 * (v @ v)
    w0, lim = _fill(S, u, sl)
    if d == 2:
        w0[:, S.modes.index((2, 0, 0))] = 1e-3 * size     # what a changed cell loses beyond its slopes
    ch = 2.0
    ref = np.any(lim(w0, ch if divb == "glm" else None) != w0, 1)
    assert ref.sum() > C // 5
    sol = Solver(3, n, d, divb, gamma=G, box_len=S.L, Mtilde=S.P.Mtilde, tvb_eps=0.0, limiter=DG_LIMIT_TVB)
    if divb == "glm":
        sol.set_glm(ch, 1.0)
    w = to_device(w0, sol)
    flags = torch.zeros(sol.stride, dtype=torch.uint8, device="cuda")
    sol.limit(w, None, flags)
    got = flags[:C].cpu().numpy().astype(bool)
    # a slope within some roundings of its limit is decided by them: leave those out
    close = np.abs(s - S.P.beta * np.minimum(dp, dm)) < 1e-12
    assert np.array_equal(got[~close], ref[~close])
