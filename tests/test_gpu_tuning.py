"""What tuning a shape does to the calls after it: those that the lane-group coder
takes keep it, a pass that runs fused uses the tuned tiling, and a tiling set by
hand is the one that runs.  The launch counters tell the two forms apart: only the
lane-group form sums in a launch of its own (accum_D1) and needs no Gram launch."""
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth

pytestmark = pytest.mark.gpu


def problem(N, p, n):
    g = torch.Generator(device="cuda:0").manual_seed(3)
    Y = sdl.signals(torch.randn(N, p, p, device="cuda:0", generator=g))
    D1, D2 = (sdl.dictionary(torch.tensor(D, dtype=torch.float32, device="cuda:0"))
              for D in synth.init_dictionaries(p, p, n, n, seed=1))
    return Y, D1, D2


def launches(ctx, fn):
    ctx.profile_collect()
    out = fn()
    assert ctx.status() == 0
    return out, {k: c for k, (_, c) in ctx.profile_collect().items()}


@pytest.mark.parametrize("p,n,s", [(8, 16, 4), (12, 24, 6), (16, 32, 8)])
def test_tuned_calls_keep_the_lane_group_coder(p, n, s):
    Y, D1, D2 = problem(200_000, p, n)
    ctx = sdl.Context(0)
    try:
        before, _ = launches(ctx, lambda: ctx.sparse_code(Y, D1, D2, s))
        _, tuning = launches(ctx, lambda: ctx.tune_tiling(Y, D1, D2, s))
        assert tuning["accum_D1"] == 0          # timing runs are not counted
        after, cnt = launches(ctx, lambda: ctx.sparse_code(Y, D1, D2, s))
        assert cnt["code"] == 1 and cnt["gram"] == 0
        for x, y in zip((before.support, before.coef, before.nnz), (after.support, after.coef, after.nnz)):
            assert torch.equal(x, y)
        # 200 000 signals: the lane groups lead by a quarter in an iteration too
        E1, E2 = D1.t().clone().t(), D2.t().clone().t()
        _, cnt = launches(ctx, lambda: ctx.iterate(Y, E1, E2, s))
        assert cnt["accum_D1"] == 1 and cnt["accum_D2"] == 1 and cnt["gram"] == 0
        # too few signals for that form: one fused launch, in the tuned tiling
        small = Y[:512]
        _, cnt = launches(ctx, lambda: ctx.iterate(small, E1, E2, s))
        assert cnt["accum_D1"] == 0 and cnt["gram"] == 1
        # a tiling set by hand runs everywhere
        ctx.set_tiling(p, p, n, n, s, sdl.tilings(p, p, n, n, s)[0])
        _, cnt = launches(ctx, lambda: ctx.sparse_code(Y, D1, D2, s))
        assert cnt["gram"] == 1
        _, cnt = launches(ctx, lambda: ctx.iterate(Y, E1, E2, s))
        assert cnt["accum_D1"] == 0 and cnt["gram"] == 1
        # unpinned again
        ctx.set_tiling(p, p, n, n, s, -1)
        _, cnt = launches(ctx, lambda: ctx.iterate(Y, E1, E2, s))
        assert cnt["accum_D1"] == 1
    finally:
        ctx.close()
