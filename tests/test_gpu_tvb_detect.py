"""The conservative detector in front of the TVB procedure must not lose a cell:
random states over weak to strong slopes, subsonic to hypersonic flow, cold gas,
and fields that are zero, aligned with an axis or generic (the degenerate
eigenvectors), for thresholds below and inside the range of the amplitudes. FP64:
the cells that change are the oracle's. FP32 form: on octree leaves of one level,
and on a list of every cell (an indicator that flags all), the state is bit for
bit that of the plain limiter on a uniform mesh, which has no detector."""
import numpy as np
import pytest

from oracle import mhd
from oracle import mlp as M
from oracle.dg import Scheme
from oracle.limiter import Limiter
from gpu_helpers import means_to_device, to_device

pytestmark = pytest.mark.gpu
G = 5.0 / 3.0
N = (11, 9, 8)


def _state(S, seed):
    r = np.random.default_rng(seed)
    C = S.C
    rho, p = np.exp(0.5 * r.normal(size=C)), np.exp(1.5 * r.normal(size=C))
    v = r.normal(size=(C, 3)) * np.exp(1.5 * r.normal(size=(C, 1)))
    B = r.normal(size=(C, 3)) * np.exp(r.normal(size=(C, 1)))
    kind = r.integers(0, 6, C)
    B[kind == 0] = 0.0
    B[kind == 1, 1:] = 0.0
    B[kind == 2] = B[kind == 2] * np.array([1.0, 1e-8, 0.0])
    u = mhd.conserved(rho, v, p, B, G)
    w = np.zeros((C, S.N))
    nleg = 9 if S.divb == "glm" else 5
    for k in range(nleg):
        mean = u[:, k] if k < 8 else 0.1 * r.normal(size=C)
        w[:, k * S.n] = mean
        w[:, k * S.n + 1:(k + 1) * S.n] = (r.normal(size=(C, S.n - 1)) * np.exp(2.0 * r.normal(size=(C, 1)))
                                           * (0.03 * np.abs(mean)[:, None] + 1e-3))
    if S.divb == "powell":
        nd = len(S.ldf)
        w[:, 5 * S.n:5 * S.n + nd] = 0.02 * r.normal(size=(C, nd)) * np.exp(2.0 * r.normal(size=(C, 1)))
        # the three constant functions: B's means (their vectors from the basis itself)
        Sv = S.Sv[5 * S.n:5 * S.n + 3, 0, 5:8]
        w[:, 5 * S.n:5 * S.n + 3] = np.linalg.solve(Sv.T, B.T).T
    return w


def _smooth(S, seed):
    """A smooth state (its slopes agree with the neighbour differences) with steeper slopes in a third of the cells."""
    r = np.random.default_rng(seed)

    def fn(x):
        t = 2 * np.pi * x
        rho = 1.0 + 0.3 * np.sin(t[..., 0] + t[..., 1])
        v = np.stack([2.0 * np.sin(t[..., 1]), np.cos(t[..., 2] + t[..., 0]), 0.5 * np.sin(t[..., 0])], -1)
        B = np.stack([0.8 + 0.2 * np.cos(t[..., 1]), 0.4 * np.sin(t[..., 2]), 0.6 * np.cos(t[..., 0])], -1)
        u = mhd.conserved(rho, v, 1.0 + 0.2 * np.cos(t[..., 2]), B, G)
        return np.concatenate([u, 0.1 * np.sin(t[..., :1])], -1) if S.V == 9 else u

    w = S.project(fn)
    hit = r.random(S.C) < 0.33
    w[hit] = np.where(S.is_mean, w[hit], w[hit] * np.exp(r.normal(size=(hit.sum(), 1))))
    return w


def _mesh(route):
    """The ragged box, or 8^3 leaves of one level in Morton order."""
    from paper_1806_02343_gb300.workloads import morton_order
    if route != "octree":
        return N, np.arange(int(np.prod(N))), dict()
    ijk = np.array([(i, j, k) for k in range(8) for j in range(8) for i in range(8)], dtype=np.int32)
    lev = np.full(512, 3, np.int8)
    order = morton_order(lev, ijk, 3, 3)
    return (8, 8, 8), order, dict(levels=lev[order], ijk=ijk[order])


@pytest.mark.parametrize("route,divb", [("fp64", "glm"), ("fp64", "powell"), ("octree", "powell"),
                                        ("listed", "glm"), ("listed", "powell")])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("mtilde", [0.01, 0.9, 5.0, 40.0, 300.0])
def test_changed_cells_are_the_oracles(route, divb, d, mtilde):
    import torch
    from paper_1806_02343_gb300.binding import DG_LIMIT_MLP, DG_LIMIT_TVB, DG_PREC_FP32MIX, DG_PREC_FP64, Solver
    n, order, tree = _mesh(route)
    fp32 = route != "fp64"
    S = Scheme(3, d, divb, G, n)
    S.P.Mtilde = mtilde
    w0 = _smooth(S, 7) if mtilde < 1.0 else _state(S, 7)
    if fp32:
        w0 = w0.astype(np.float32).astype(np.float64)
    ch = 3.0

    def limit(limiter, order, **kw):
        sol = Solver(3, None if "levels" in kw else n, d, divb, gamma=G, box_len=S.L, Mtilde=mtilde, limiter=limiter,
                     precision=DG_PREC_FP32MIX if fp32 else DG_PREC_FP64, **kw)
        if divb == "glm":
            sol.set_glm(ch, 1.0)
        if limiter == DG_LIMIT_MLP:
            theta = np.zeros_like(M.init_params(sol.n_features(), seed=1))
            theta[-1] = 1.0  # the output's bias: every cell's probability is above one half
            sol.mlp_set_weights(torch.as_tensor(theta, dtype=torch.float32, device="cuda"), 0.5)
        w = to_device(w0[order], sol)
        flags = torch.zeros(sol.stride, dtype=torch.uint8, device="cuda")
        sol.limit(w, means_to_device(w0[order], sol, S) if fp32 else None, flags)
        hit = flags[: sol.ncell].cpu().numpy().astype(bool)
        assert sol.limiter_counts()["limited"] == hit.sum()
        return hit, w[:, : sol.ncell].cpu().numpy()

    hit, w = limit(DG_LIMIT_MLP if route == "listed" else DG_LIMIT_TVB, order, **tree)
    if fp32:
        ref, wr = limit(DG_LIMIT_TVB, np.arange(S.C))
        assert np.array_equal(w, wr[:, order])
    else:
        ref = np.any(Limiter(S, tvb=True, positivity=False)(w0, ch if divb == "glm" else None) != w0, 1)
    assert ref.any()
    assert np.array_equal(hit, ref[order])
