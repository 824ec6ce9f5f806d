"""Small solves: walks one per lane, summed per point afterwards (walk_sum_kernel), against the
per-walk estimates of the same walks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _ctx():
    import paper_2201_13240_gb300 as wos
    return wos.Context(0)


@pytest.mark.parametrize("npts,walks", [(1, 1), (1, 31), (1, 33), (2, 64), (1, 129), (130, 1), (43, 3), (5, 77),
                                        (8192, 128), (8193, 128)])
@pytest.mark.parametrize("kind", ["plain2d", "plain3d", "window", "mesh"])
def test_sums_equal_the_walks(kind, npts, walks):
    """Counts are exact.  A lane adds at most 128 walks of a point in FP32: its rounding is at most
    128 * 2^-24 of the sum of magnitudes (and of squares); the estimates themselves are the same."""
    import torch
    if kind == "mesh" and npts * walks > 4096:
        pytest.skip("the mesh walk's small solves take the same summation")
    ctx = _ctx()
    desc, eps = {"plain2d": (W.square2d_problem, 1e-3), "plain3d": (W.cube3d_problem, 1e-4),
                 "window": (W.hifreq_alpha_problem, 1e-3),
                 "mesh": (lambda: W.mesh_manufactured_problem(level=2), 1e-4)}[kind]
    desc = desc()
    prob = ctx.problem(desc)
    sb = ctx.sigma_bar(prob, 32)[0]
    pts = W.mesh_interior_points(npts, 5) if kind == "mesh" else W.uniform_in_box(desc["dim"], npts, 0.02, 0.98, 5)
    pts = torch.from_numpy(pts).cuda()
    window = (0.5, 1.5) if kind == "window" else None
    (s, s2, n), st = ctx.solve(prob, pts, walks, eps, sb, seed=7, walk_offset=3, window=window)
    u, k, st1 = ctx.walk_estimates(prob, pts, walks, eps, sb, seed=7, walk_offset=3, window=window)
    assert torch.all(n == walks)
    assert torch.equal(st, st1)
    tol = 128 * 2.0 ** -24
    assert torch.all((s - u.sum(1)).abs() <= tol * u.abs().sum(1))
    # the partial sums are shifted by a walk's value c: (u - c)^2 and 2 c (u - c) are rounded, each
    # at most 4 max u^2
    big = u.abs().max(1).values ** 2 * walks
    assert torch.all((s2 - u.square().sum(1)).abs() <= 8 * tol * big)
