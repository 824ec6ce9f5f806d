"""Gradient walks of B-spline fields in generic and compiled kernels."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_compiled_gradient_walks_part_no_more_than_plain_ones():
    """Both gradient kernels of B-spline fields name the same rounding of the Green's function, so a walk in
    the compiled kernel parts from its twin in the generic one only where the fields' roundings differ,
    which the plain walks show: the shares of equal estimates agree to 0.008 (three standard errors of
    a share of 0.96 over 51,200 walks on each side, 0.0026 each, and the first ball's further terms)."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    desc = W.noise_cube_problem()
    generic, compiled = ctx.problem(desc), ctx.problem(desc)
    compiled.specialize(("fp32",), ("plain", "grad"))
    pts = torch.from_numpy(W.uniform_in_box(3, 800, 0.02, 0.98, 3)).cuda()
    sb = ctx.sigma_bar(generic, 32)[0]

    def equal(f):
        a, b = f(generic, pts, 64, 1e-4, sb, seed=5)[0], f(compiled, pts, 64, 1e-4, sb, seed=5)[0]
        return float((a == b).double().mean())
    assert equal(ctx.walk_grad_estimates) >= equal(ctx.walk_estimates) - 0.008
