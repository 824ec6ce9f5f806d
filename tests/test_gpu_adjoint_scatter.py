"""The adjoint's warp-wide scatter and its joint call: grids at the edges of the shared-memory copy,
2D and 3D, points in clamped cells."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _problem(dim, ares):
    lo, hi = [0.0] * dim, [1.0] * dim
    rng = np.random.default_rng(sum(ares))
    grid = lambda res, a, b: rng.uniform(a, b, res[::-1]).astype(np.float32)
    g = W.sst(W.term(1.0), W.term(1.0, (W.LIN, 1.0, 0.0)))
    return W.problem(dim, W.box(lo, hi), W.grid_field("grid_bspline", grid(ares, 0.8, 1.25), lo, hi),
                     W.grid_field("grid_linear", grid([5] * dim, 0.0, 4.0), lo, hi), W.const(1.0), g)


@pytest.mark.parametrize("ares", [[4, 4], [5, 9], [64, 128], [65, 127], [4, 4, 4], [7, 5, 6], [16, 16, 32],
                                  [17, 16, 32], [5, 5, 327]])
@pytest.mark.parametrize("npts,walks", [(1, 1), (37, 3)])
def test_fp32_gradients_equal_fp64(ares, npts, walks):
    """FP32 against FP64 replays of the same walks (uniforms differ by 2^-24, so a walk may part from
    its FP64 twin: the gradients agree to 5e-2, as in the adjoint's other FP32 test), each call's
    gradient against the joint call's (1e-5: FP32 sums in another order), and the joint call's
    statistics, which count each gradient's replay."""
    import torch

    import paper_2201_13240_gb300 as wos
    dim = len(ares)
    ctx = wos.Context(0)
    prob = ctx.problem(_problem(dim, ares))
    pts = torch.from_numpy(W.uniform_in_box(dim, npts, 0.02, 0.98, 8)).cuda()
    gu = torch.linspace(0.5, 1.5, npts, dtype=torch.float64, device="cuda")
    ns, na = 5 ** dim, int(np.prod(ares))
    out = {}
    for prec in ("fp32", "fp64"):
        gs = torch.zeros(ns, dtype=torch.float64, device="cuda")
        ga = torch.zeros(na, dtype=torch.float64, device="cuda")
        s1, s2, s3 = ctx.new_stats(), ctx.new_stats(), ctx.new_stats()
        ctx.adjoint_sigma(prob, pts, walks, gu, gs, 1e-3, 60.0, seed=2, precision=prec, stats=s1)
        ctx.adjoint_alpha(prob, pts, walks, gu, ga, 1e-3, 60.0, seed=2, precision=prec, stats=s2)
        js, ja = ctx.adjoint(prob, pts, walks, 1e-3, 60.0, gu, ns, na, seed=2, precision=prec, stats=s3)
        assert torch.equal(s1 + s2, s3) and int(s1[1]) == npts * walks
        for one, joint in ((gs, js), (ga, ja)):
            assert torch.isfinite(one).all()
            assert (one - joint).norm() <= 1e-5 * one.norm()
        out[prec] = (gs, ga)
    if dim == 3:  # the 3D uniforms are the same in both precisions
        for a, b in zip(out["fp32"], out["fp64"]):
            assert (a - b).norm() <= 5e-2 * b.norm()
