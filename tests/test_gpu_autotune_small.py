"""The batch autotuner on batches of at most 2^20 walks."""
import time

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nprob,points", [(4, 256), (8, 512)])
def test_tuned_small_batches_are_no_slower(nprob, points):
    """The default schedule of so small a batch runs one walk per lane, and its trial does too: what the
    tuner keeps is at most 8 % slower than the default (medians of 60 solves; a set chunk, which trials on
    the large solves' path preferred, was 13 to 17 % slower).  Estimates stay the same walks."""
    import torch

    import paper_2201_13240_gb300 as wos
    ctx = wos.Context(0)
    probs, pts, offs, walks = W.batch_problems(nprob, seed=7, max_points=points, max_walks=128)
    assert walks.sum() <= 1 << 20
    hp = [ctx.problem(q) for q in probs]
    batch = ctx.batch(hp, offs, [ctx.sigma_bar(h, 64)[0] for h in hp])
    pts, walks = torch.from_numpy(pts).cuda(), torch.from_numpy(walks).cuda()

    def median():
        t = []
        for _ in range(60):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            acc, _ = ctx.solve_batch(batch, pts, walks, 1e-3, seed=3)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return sorted(t)[30], acc
    median()
    default, a = median()
    best, best_ms, default_ms = ctx.batch_autotune(batch, pts, walks, 1e-3, seed=3, trial_shift=0)
    assert 0 < best_ms <= default_ms
    tuned, b = median()
    assert tuned <= 1.08 * default, (best, tuned, default)
    assert torch.equal(a[2], b[2]) and torch.allclose(a[0], b[0], rtol=1e-4)
