"""Event timing covers the kernel that runs, whichever form a call takes: one record
per launch, around that launch."""
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(20, 20), (48, 20), (20, 48)])   # 48: past the lane kernel's 32 atoms
def test_update_time_holds_the_accumulation(n1, n2):
    N, p, s = 400_000, 16, 4
    g = torch.Generator(device="cuda:0").manual_seed(1)
    Y = sdl.signals(torch.randn(N, p, p, device="cuda:0", generator=g))
    D1, D2 = (sdl.dictionary(torch.tensor(D, dtype=torch.float32, device="cuda:0"))
              for D in synth.init_dictionaries(p, p, n1, n2, seed=1))
    q = torch.randint(0, n1 * n2, (N, s), device="cuda:0", generator=g, dtype=torch.int32)
    codes = sdl.Codes(q, torch.randn(N, s, device="cuda:0", generator=g), None)
    ctx = sdl.Context(0)
    try:
        ctx.update_D1(Y, D1, D2, codes)
        ctx.update_D2(Y, D1, D2, codes)
        ctx.profile()
        ctx.profile_collect()
        ctx.update_D1(Y, D1, D2, codes)
        ctx.update_D2(Y, D1, D2, codes)
        prof = ctx.profile_collect()
        assert ctx.status() == 0
        # each side reads the 410 MB of signals, more than L2 holds: 51 us at 8 TB/s
        for k in ("accum_D1", "accum_D2"):
            ms, count = prof[k]
            assert count == 1 and ms > 0.05, (k, ms)
    finally:
        ctx.close()


@pytest.mark.parametrize("p,n,s", [((4, 4, 4), (8, 8, 8), 4), ((4, 4, 5), (6, 6, 7), 4)])
def test_three_mode_coding_counts_one_launch(p, n, s):
    g = torch.Generator(device="cuda:0").manual_seed(1)
    Y = sdl.signals3(torch.randn(500, *p, device="cuda:0", generator=g))
    D = [torch.randn(a, b, device="cuda:0", generator=g) for a, b in zip(p, n)]
    D = [sdl.dictionary(d / d.norm(dim=0)) for d in D]
    ctx = sdl.Context(0)
    try:
        ctx.profile()
        ctx.sparse_code3(Y, *D, s)
        prof = ctx.profile_collect()
        assert ctx.status() == 0
        assert prof["code"][1] == 1 and prof["code"][0] > 0
    finally:
        ctx.close()
