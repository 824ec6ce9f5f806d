"""Solves with per-point walk counts on both sides of the small-solve limit (2^20 walks), in compiled
kernels of every kind of fields, in generic ones and in batches: counts are exact, the sums are those
of the walks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
LIMIT = 1 << 20


def _counts(npts, total, rng):
    """Walks per point, runs of points without walks among them, with the given sum."""
    c = rng.multinomial(total, rng.dirichlet(np.ones(npts) * 4)).astype(np.int32)
    c[npts // 3:npts // 3 + 5] = 0
    c[-1] = 0
    c[0] += total - c.sum()
    return c


@pytest.mark.parametrize("total", [1, 900, LIMIT, LIMIT + 1])
@pytest.mark.parametrize("kind,spec", [("square2d", True), ("noise_annulus", True), ("noise_cube", True),
                                       ("hifreq", True), ("square2d", False), ("noise_cube", False),
                                       ("hifreq", False)])
def test_per_point_counts_sum_the_walks(kind, spec, total):
    """A lane adds n consecutive walks of a point in FP32, at most all of them: the rounding is at most
    n * 2^-24 of the sum of magnitudes, and for the squares (shifted by a walk's value) 8 n * 2^-24 of
    n max u^2, on points where those squares stay in FP32's range: 2 max |u| < 2^63).  walk_offset != 0,
    and the kernel's own per-walk estimates of the same walks."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    desc = {"square2d": W.square2d_problem, "noise_annulus": W.noise_annulus_problem, "noise_cube": W.noise_cube_problem,
            "hifreq": W.hifreq_alpha_problem}[kind]()
    window = (0.5, 1.5) if kind == "hifreq" else None
    prob = ctx.problem(desc)
    if spec:
        prob.specialize(("fp32",), ("window" if window else "plain",))
    npts, rng = 700, np.random.default_rng(total % 97)
    counts = _counts(npts, total, rng)
    assert counts.sum() == total and counts.min() == 0
    r, t = np.sqrt(rng.uniform(0.4 ** 2, 1.05 ** 2, npts)), rng.uniform(0, 2 * np.pi, npts)
    pts = np.stack([r * np.cos(t), r * np.sin(t)]).astype(np.float32) if kind == "noise_annulus" else \
        W.uniform_in_box(desc["dim"], npts, 0.02, 0.98, 5)
    pts = torch.from_numpy(pts).cuda()
    most = int(counts.max())
    (s, s2, n), st = ctx.solve(prob, pts, torch.from_numpy(counts).cuda(), 1e-3, 50.0, seed=7, walk_offset=5, window=window)
    u, _, _ = ctx.walk_estimates(prob, pts, most, 1e-3, 50.0, seed=7, walk_offset=5, window=window)
    assert np.array_equal(n.cpu().numpy(), counts) and int(st[1]) == total
    u = torch.where(torch.arange(most, device="cuda")[None, :] < torch.from_numpy(counts).cuda()[:, None], u, 0.0)
    tol = max(128, most) * 2.0 ** -24
    assert torch.all((s - u.sum(1)).abs() <= tol * u.abs().sum(1))
    big = u.abs().max(1).values
    fits = 2 * big < 2.0 ** 63
    assert fits.any()
    assert torch.all(((s2 - u.square().sum(1)).abs() <= 8 * tol * big ** 2 * n)[fits])


@pytest.mark.parametrize("spec", [True, False])
@pytest.mark.parametrize("per_point", [0, 1, 40, 3000])
def test_batches_sum_the_same_walks_on_either_path(spec, per_point):
    """A batch on the kernel's own schedule, which spreads at most 2^20 walks, against the same kernel
    with a set chunk, which never does: the same walks, so counts and statistics are equal and the sums
    differ by the rounding of a point's FP32 sums (as above).  per_point = 0: the batch's own counts."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    probs, pts, offs, walks = W.batch_problems(9, seed=5, max_points=90, max_walks=200)
    hp = [ctx.problem(q) for q in probs]
    batch = ctx.batch(hp, offs, [ctx.sigma_bar(h, 32)[0] for h in hp])
    if spec:
        batch.specialize(("fp32",))
    pts = torch.from_numpy(pts).cuda()
    walks = walks.copy() if per_point == 0 else np.full(pts.shape[1], per_point, np.int32)
    walks[::7] = 0
    w = torch.from_numpy(walks).cuda()
    out = []
    for chunk in (0, 64):
        batch.set_schedule(chunk=chunk)
        out.append(ctx.solve_batch(batch, pts, w, 1e-3, seed=3, walk_offset=2))
    ((s, s2, n), st), ((r, r2, m), rt) = out
    assert torch.equal(n, m) and torch.equal(st, rt) and np.array_equal(n.cpu().numpy(), walks)
    tol = 2 * max(128, int(walks.max())) * 2.0 ** -24
    rms = (r2 * m).sqrt()  # at least the sum of magnitudes
    assert torch.all((s - r).abs() <= tol * rms)
    assert torch.all((s2 - r2).abs() <= 8 * tol * r2 * m)


@pytest.mark.parametrize("kind", ["square2d", "cube3d", "noise_annulus", "noise_cube", "hifreq"])
def test_forms_of_the_generic_kernel_round_alike(kind):
    """One walk per point: its sum is its estimate, a product of two FP32 numbers and so exact in FP64, in the
    form that writes estimates, in the small solves' form and in the form of per-point counts."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    desc = {"square2d": W.square2d_problem, "cube3d": W.cube3d_problem, "noise_annulus": W.noise_annulus_problem,
            "noise_cube": W.noise_cube_problem, "hifreq": W.hifreq_alpha_problem}[kind]()
    prob = ctx.problem(desc)
    sb = ctx.sigma_bar(prob, 32)[0]
    n, rng = 3000, np.random.default_rng(2)
    r, t = np.sqrt(rng.uniform(0.4 ** 2, 1.05 ** 2, n)), rng.uniform(0, 2 * np.pi, n)
    pts = np.stack([r * np.cos(t), r * np.sin(t)]).astype(np.float32) if kind == "noise_annulus" else \
        W.uniform_in_box(desc["dim"], n, 0.02, 0.98, 5)
    pts, ones = torch.from_numpy(pts).cuda(), torch.ones(n, dtype=torch.int32, device="cuda")
    for window in (None, (0.5, 1.5)):
        u = ctx.walk_estimates(prob, pts, 1, 1e-3, sb, seed=9, window=window)[0][:, 0]
        for walks in (1, ones):
            (s, s2, _), _ = ctx.solve(prob, pts, walks, 1e-3, sb, seed=9, window=window)
            assert torch.equal(s, u)
            assert torch.allclose(s2, u * u, rtol=1e-15, atol=0)
