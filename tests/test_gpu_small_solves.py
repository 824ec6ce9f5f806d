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


@pytest.mark.parametrize("most", [1, 3, 200, 5000])
def test_per_point_counts(most):
    """Walks per point from 0 up (runs of points without walks among them): counts are exact, and the
    sums are those of the walks' own estimates (rounding as above, with at most `most` walks of a
    point in a lane); most = 5000 is above the small-solve limit of 2^20 walks."""
    import torch
    ctx = _ctx()
    prob = ctx.problem(W.square2d_problem())
    npts = 700
    pts = torch.from_numpy(W.uniform_in_box(2, npts, 0.02, 0.98, 5)).cuda()
    rng = np.random.default_rng(most)
    counts = rng.integers(0, most + 1, npts).astype(np.int32)
    counts[100:400:1 if most == 1 else 7] = 0
    counts[-1] = 0
    (s, s2, n), st = ctx.solve(prob, pts, torch.from_numpy(counts).cuda(), 1e-3, 50.0, seed=7)
    assert np.array_equal(n.cpu().numpy(), counts) and int(st[1]) == int(counts.sum())
    u, _, _ = ctx.walk_estimates(prob, pts, most, 1e-3, 50.0, seed=7)
    u = torch.where(torch.arange(most, device="cuda")[None, :] < torch.from_numpy(counts).cuda()[:, None], u, 0.0)
    tol = max(128, most) * 2.0 ** -24
    assert torch.all((s - u.sum(1)).abs() <= tol * u.abs().sum(1))


@pytest.mark.parametrize("kind", ["square2d", "cube3d", "noise_cube", "noise_annulus"])
def test_register_variants_walk_the_same_walks(kind):
    """The generic kernel's variants (by fields, and above 2^20 walks) run the same arithmetic."""
    import torch
    ctx = _ctx()
    desc = {"square2d": W.square2d_problem, "cube3d": W.cube3d_problem, "noise_cube": W.noise_cube_problem,
            "noise_annulus": W.noise_annulus_problem}[kind]()
    prob = ctx.problem(desc)
    rng = np.random.default_rng(1)
    n = 64
    r, t = np.sqrt(rng.uniform(0.4 ** 2, 1.05 ** 2, n)), rng.uniform(0, 2 * np.pi, n)
    pts = np.stack([r * np.cos(t), r * np.sin(t)]).astype(np.float32) if kind == "noise_annulus" else \
        W.uniform_in_box(desc["dim"], n, 0.05, 0.95, 2)
    pts = torch.from_numpy(pts).cuda()
    many = (1 << 20) // n + 1
    a, ka, _ = ctx.walk_estimates(prob, pts, 50, 1e-3, 40.0, seed=3)
    b, kb, _ = ctx.walk_estimates(prob, pts, many, 1e-3, 40.0, seed=3)
    assert torch.equal(a, b[:, :50]) and torch.equal(ka, kb[:, :50])
