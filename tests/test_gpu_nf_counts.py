"""Next-flight solves with per-point walk counts, on both sides of the limit where another register cap
takes over: the sums are those of the walks, whichever of the two launches ran them."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("terms", [0, 8])
@pytest.mark.parametrize("kind,few", [("square2d", 1 << 18), ("cube3d", 1 << 18), ("noise_cube", 1 << 20), ("mesh", 3 << 18)])
@pytest.mark.parametrize("over", [None, 0, 1])
def test_sums_equal_the_walks(kind, few, terms, over):
    """over: walks above the limit (None: a handful).  Estimates are added in FP64: the sums agree with the
    per-walk estimates' to 1e-12 of the sum of magnitudes (of squares), counts exactly; the estimates'
    launch has its own size, so its register cap may be the other one."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    desc = {"square2d": W.square2d_problem, "cube3d": W.cube3d_problem, "noise_cube": W.noise_cube_problem,
            "mesh": lambda: W.mesh_manufactured_problem(level=2, tol=0.25)}[kind]()
    prob = ctx.problem(desc)
    sb = ctx.sigma_bar(prob, 32)[0]
    npts, rng = 2048, np.random.default_rng(7)
    total = 501 if over is None else few + over
    counts = rng.multinomial(total, rng.dirichlet(np.full(npts, 50.0))).astype(np.int32)
    counts[1] += counts[5]
    counts[5] = 0
    most = int(counts.max())
    pts = W.mesh_interior_points(npts, 5) if kind == "mesh" else W.uniform_in_box(desc["dim"], npts, 0.02, 0.98, 5)
    pts = torch.from_numpy(pts).cuda()
    (s, s2, n), st = ctx.solve_nf(prob, pts, torch.from_numpy(counts).cuda(), 1e-3, sb, seed=7, series_terms=terms)
    u, _, _ = ctx.walk_estimates_nf(prob, pts, most, 1e-3, sb, seed=7, series_terms=terms)
    assert np.array_equal(n.cpu().numpy(), counts) and int(st[1]) == total
    u = torch.where(torch.arange(most, device="cuda")[None, :] < torch.from_numpy(counts).cuda()[:, None], u, 0.0)
    assert torch.all((s - u.sum(1)).abs() <= 1e-12 * u.abs().sum(1))
    assert torch.all((s2 - u.square().sum(1)).abs() <= 1e-12 * u.square().sum(1))
