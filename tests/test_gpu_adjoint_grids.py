"""The alpha gradient on 2D and non-cubic 3D control grids, on both sides of the per-CTA copy's limit
and with thin grids, against the oracle's central differences on the same walks."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _problem(dim, ares, alpha):
    lo, hi = [0.0] * dim, [1.0] * dim
    sig = np.random.default_rng(dim).uniform(0.0, 4.0, [5] * dim).astype(np.float32)
    g = W.sst(W.term(1.0), W.term(1.0, (W.LIN, 1.0, 0.0)))
    return W.problem(dim, W.box(lo, hi), W.grid_field("grid_bspline", alpha, lo, hi),
                     W.grid_field("grid_linear", sig, lo, hi), W.const(1.0), g)


def _alpha(ares):
    """A smooth field's values as controls, so that sigma' keeps the size of the problem's own terms."""
    ax = [np.linspace(0.0, 1.0, n) for n in ares[::-1]]
    grid = np.meshgrid(*ax, indexing="ij")
    return (1.0 + 0.2 * np.sin(2.0 * sum((i + 1) * c for i, c in enumerate(grid)))).astype(np.float32)


@pytest.mark.parametrize("ares", [[16, 12], [5, 40], [64, 128], [96, 100], [5, 9, 7], [4, 4, 40], [16, 16, 32], [24, 20, 18]])
def test_alpha_gradient_equals_the_oracles_differences(orc, ares):
    """FP64 replays.  A control's step h moves sigma' by up to h / spacing^2 <= 1e4 h, some hundred times h
    relative to sigma_bar, on the few steps of a walk in its support: the difference quotient is off by the
    square of that, (1e-6 * 1e3)^2 = 1e-6 at most, and by 1e-16 / h = 1e-10 of the mean: 1e-5 of the gradient
    (of its largest entry's thousandth where a control's own is smaller).  Among the controls are corners,
    which points in the boundary cells reach through clamped indices."""
    import torch

    import paper_2201_13240_gb300 as wos
    dim, alpha = len(ares), _alpha(ares)
    desc = _problem(dim, ares, alpha)
    sb = orc.sigma_bar(desc, 24)[0]
    pts = np.concatenate([W.uniform_in_box(dim, 9, 0.05, 0.95, 4), np.full((dim, 1), 0.01, np.float32),
                          np.full((dim, 1), 0.99, np.float32)], 1).astype(np.float32)
    gu = np.random.default_rng(3).normal(size=pts.shape[1])
    walks, seed, eps, h = 8, 5, 1e-3, 1e-6
    ctx = wos.Context(0)
    prob = ctx.problem(desc)
    grad = torch.zeros(alpha.size, dtype=torch.float64, device="cuda")
    ctx.adjoint_alpha(prob, torch.from_numpy(pts).cuda(), walks, torch.from_numpy(gu).cuda(), grad, eps, sb, seed=seed,
                      precision="fp64")
    g = grad.cpu().numpy()
    assert np.isfinite(g).all()
    order = np.argsort(-np.abs(g))
    for node in [0, alpha.size - 1, ares[0] - 1, *order[[0, 1, 5, 20, 60]]]:
        val, at = [], []
        for s in (1, -1):
            a = alpha.copy().reshape(-1)
            a[node] += np.float32(s * h)
            at.append(float(a[node]))
            u, _ = orc.walks(_problem(dim, ares, a.reshape(alpha.shape)), pts, walks, seed=seed, eps=eps, sigma_bar=sb)
            val.append((gu * u.mean(axis=1)).sum())
        fd = (val[0] - val[1]) / (at[0] - at[1])
        assert abs(g[node] - fd) <= 1e-5 * max(abs(fd), 1e-3 * np.abs(g).max()), (node, g[node], fd)
