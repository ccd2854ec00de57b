"""Contexts that live side by side share the kernels' constant tables: a Powell
context's timestep and step are bit for bit the same whether or not other contexts
of the same degree and precision (either scheme, uniform or octree) were created
after it."""
import numpy as np
import pytest

from test_gpu_sf import _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("mesh", ["uniform", "octree"])
@pytest.mark.parametrize("other", ["glm", "powell"])
def test_a_powell_context_is_not_changed_by_others(d, prec, mesh, other):
    import torch
    from paper_1806_02343_gb300.binding import DG_PREC_FP32MIX, DG_PREC_FP64, Solver
    p = dict(precision=DG_PREC_FP32MIX if prec == "fp32" else DG_PREC_FP64)
    n, tree = (8, 8, 8), {}
    if mesh == "octree":
        ijk = np.array([(i, j, k) for k in range(8) for j in range(8) for i in range(8)], dtype=np.int32)
        n, tree = None, dict(levels=np.full(512, 3, np.int8), ijk=ijk)
    outs = []
    for disturb in (False, True):
        sol = Solver(3, n, d, "powell", **tree, **p)
        w = _state(sol, 3).to(sol.dtype)
        wm = w[sol.mean_rows()].double().contiguous() if sol.fp32 else None
        if disturb:
            Solver(3, (6, 5, 4), d, other, **p)
        dt = sol.dt(w, wm)
        sol.step(w, wm)
        assert sol.status() == 0
        outs.append([dt.cpu().numpy(), w.cpu().numpy()] + ([wm.cpu().numpy()] if sol.fp32 else []))
    for a, b in zip(*outs):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)
