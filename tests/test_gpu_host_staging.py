"""wos_solve_host's page-locked results: a small call takes them also after a large one on the context."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _copies(call):
    """Copies to the host during a call, by the kind of host memory, as the profiler names them."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):  # a process's first session may see nothing
        torch.zeros(8, device="cuda").cpu()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        out = call()
    names = [e.name for e in p.events()]
    if not any("DtoH" in n for n in names):
        pytest.skip("the profiler reports no copies here")
    return out, sum("DtoH" in n and "Pinned" in n for n in names), sum("DtoH" in n and "Pageable" in n for n in names)


def test_small_calls_stay_staged_after_a_large_one():
    import torch

    import paper_2201_13240_gb300 as wos
    ctx, fresh = wos.Context(0), wos.Context(0)
    prob, twin = ctx.problem(W.square2d_problem()), fresh.problem(W.square2d_problem())
    small, large = W.uniform_in_box(2, 1000, 0.02, 0.98, 1), W.uniform_in_box(2, 70000, 0.02, 0.98, 1)
    solve = lambda c, p, pts: c.solve_host(p, pts, 2, 1e-3, 40.0, seed=3)
    solve(ctx, prob, small)
    _, pinned, pageable = _copies(lambda: solve(ctx, prob, large))
    assert pinned == 0 and pageable == 4
    got, pinned, pageable = _copies(lambda: solve(ctx, prob, small))
    assert pinned == 2 and pageable == 0
    want = solve(fresh, twin, small)
    assert all(torch.allclose(a, b, rtol=1e-9, atol=1e-9) for a, b in zip(got[:3], want[:3])) and torch.equal(got[3], want[3])


@pytest.mark.parametrize("npts", [1, 12288, 12289, 70000])
def test_results_equal_the_device_solve(npts):
    """The same walks on either side of the staging limit; sums that meet in atomics in another order round
    in FP64 (1e-16 each, 1e-9 allows for the variance's cancellation)."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    prob = ctx.problem(W.square2d_problem())
    pts = W.uniform_in_box(2, npts, 0.02, 0.98, 1)
    mean, var, se, st = ctx.solve_host(prob, pts, 3, 1e-3, 40.0, seed=3)
    acc, dst = ctx.solve(prob, torch.from_numpy(pts).cuda(), 3, 1e-3, 40.0, seed=3)
    for a, b in zip((mean, var, se), ctx.finalize(acc)):
        assert torch.allclose(a, b.cpu(), rtol=1e-9, atol=1e-9, equal_nan=True)
    assert torch.equal(st, dst.cpu())
