"""Cold streams in FP64: zero pressure and field, one velocity, densities that
differ from cell to cell. All waves of a face move with the stream, and the flux
is the upwind side's, in every direction the stream can take across the axes. The
specialised kernels against the generic ones (generic_kernels = 1): finite, and
equal to some hundred roundings."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(3, "glm", 1), (3, "glm", 2), (3, "glm", 3), (3, "powell", 1), (3, "powell", 2)] + \
        [(2, s, d) for s in ("glm", "powell") for d in (1, 2, 3)]


@pytest.mark.parametrize("dim,divb,degree", CASES)
def test_cold_stream(dim, divb, degree):
    import torch
    from paper_1806_02343_gb300.binding import Solver
    n = (6, 5, 4)[:dim]
    for sx, sy, sz in itertools.product((1.0, -1.0), repeat=3):
        outs = []
        for generic in (0, 1):
            sol = Solver(dim, n, degree, divb, generic_kernels=generic)
            if divb == "glm":
                sol.set_glm(2.0, 1.0)
            w = np.zeros((sol.nrows, sol.stride))
            rho = np.random.default_rng(7).choice([1.0, 2.0, 4.0], sol.stride)
            for row, f in zip(sol.mean_rows(), (1.0, sx, 2.0 * sy, sz, 3.0)):  # E = rho v^2 / 2: p = 0 exactly
                w[row] = f * rho
            w = torch.as_tensor(w, device="cuda")
            out = torch.zeros_like(w)
            sol.rhs(w, None, out)
            outs.append(out[:, : sol.ncell].cpu().numpy())
        a, b = outs
        assert np.all(np.isfinite(b)) and np.max(np.abs(b)) > 1.0
        assert np.all(np.isfinite(a)) and np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
