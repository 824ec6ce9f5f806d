"""The mesh walk's shared leaf tests: leaves of any size, warps with few walks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies", [2, 6])
@pytest.mark.parametrize("npts,walks", [(1, 1), (3, 5), (33, 4), (700, 3)])
def test_duplicated_triangles_change_nothing(copies, npts, walks):
    """Every triangle several times over (leaves of up to four of them, and longer ones where the
    hierarchy cannot split copies): with exact radii the distances and closest points are the
    same numbers, so every walk is the same walk."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    one = W.mesh_manufactured_problem(level=2)
    many = dict(one, domain=dict(one["domain"], tris=np.repeat(one["domain"]["tris"], copies, axis=0)))
    pts = torch.from_numpy(W.mesh_interior_points(npts, 9)).cuda()
    a, b = ctx.problem(one), ctx.problem(many)
    sb = ctx.sigma_bar(a, 32)[0]
    ua, ka, sa = ctx.walk_estimates(a, pts, walks, 1e-4, sb, seed=4)
    ub, kb, st = ctx.walk_estimates(b, pts, walks, 1e-4, sb, seed=4)
    assert torch.equal(ua, ub) and torch.equal(ka, kb)
    assert int(sa[1]) == npts * walks and int(st[8]) == 0
