"""Octree set-up on several host threads (meshes of two or more parts of 8192
leaves): the face lists equal a leaf-by-leaf search, and on the GPU a context on
32^3 leaves of one level gives the residual and the limited state of the uniform
mesh (face entries, renumbered faces, side lists)."""
import itertools

import numpy as np
import pytest

from paper_1806_02343_gb300.workloads import morton_order


def _mesh():
    """16^3 cells, those of a slab refined, some of the children again: levels 4 to 6."""
    leaves = []
    for k in itertools.product(range(16), repeat=3):
        if not 3 <= k[0] < 13:
            leaves.append((4, k))
            continue
        for o in itertools.product((0, 1), repeat=3):
            c = tuple(2 * a + b for a, b in zip(k, o))
            if c[0] in range(12, 18) and c[1] < 16:
                leaves += [(6, tuple(2 * a + b for a, b in zip(c, p))) for p in itertools.product((0, 1), repeat=3)]
            else:
                leaves.append((5, c))
    lev = np.array([l for l, _ in leaves], np.int8)
    ijk = np.array([k for _, k in leaves], np.int32)
    order = morton_order(lev, ijk, 3, 6)
    return lev[order], ijk[order]


@pytest.mark.parametrize("shuffled", [False, True])
def test_faces_of_many_parts(shuffled):
    from paper_1806_02343_gb300.binding import octree_faces
    lev, ijk = _mesh()
    if shuffled:
        o = np.random.default_rng(0).permutation(len(lev))
        lev, ijk = lev[o], ijk[o]
    assert len(lev) > 4 * 8192
    at = {(int(l), *map(int, k)): i for i, (l, k) in enumerate(zip(lev, ijk))}
    want = []
    for i, (l, k) in enumerate(zip(lev.tolist(), ijk.tolist())):
        for a in range(3):
            others = [b for b in range(3) if b != a]
            for s in (-1, 1):
                nk = list(k)
                nk[a] = (nk[a] + s) % (1 << l)
                j = at.get((l, *nk))
                if j is not None:
                    if s < 0:
                        want.append((j, i, a))
                    continue
                j = at.get((l - 1, *(x >> 1 for x in nk)))
                if j is not None:
                    sub = sum((k[b] & 1) << q for q, b in enumerate(others))
                    want.append((j, i, a | 4 | sub << 4) if s < 0 else (i, j, a | 8 | sub << 4))
    got = np.stack(octree_faces(lev, ijk), 1)
    assert np.array_equal(got, np.array(want, np.int32))


@pytest.mark.gpu
@pytest.mark.parametrize("degree", [1, 2])
def test_context_equals_the_uniform_mesh(degree):
    import torch
    from paper_1806_02343_gb300.binding import DG_LIMIT_TVB, Solver
    n = 32
    ijk = np.array([(i, j, k) for k in range(n) for j in range(n) for i in range(n)], np.int32)
    lev = np.full(n ** 3, 5, np.int8)
    order = morton_order(lev, ijk, 3, 5)
    r = np.random.default_rng(2)
    out = []
    for tree in (False, True):
        kw = dict(levels=lev[order], ijk=ijk[order]) if tree else {}
        sol = Solver(3, None if tree else (n, n, n), degree, "powell", limiter=DG_LIMIT_TVB, **kw)
        if not tree:
            w0 = 0.02 * r.standard_normal((sol.nrows, sol.ncell))
            for row, m in zip(sol.mean_rows(), [1.2, 0.3, -0.2, 0.4, 3.0, 0.5, -0.4, 0.3]):
                w0[row] = m * (1.0 + 0.1 * r.standard_normal(sol.ncell))
        w = torch.zeros((sol.nrows, sol.stride), dtype=torch.float64, device="cuda")
        w[:, : sol.ncell] = torch.as_tensor(w0[:, order] if tree else w0, device="cuda")
        rhs = torch.zeros_like(w)
        sol.rhs(w, None, rhs)
        sol.limit(w, None)
        out.append([x[:, : sol.ncell].cpu().numpy() for x in (rhs, w)])
    for a, b in zip(*out):
        assert np.max(np.abs(a[:, order] - b)) <= 1e-12 * np.max(np.abs(a))  # another order of the sums, some hundred roundings
