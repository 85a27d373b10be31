"""Error-driven code-only batches on both sides of their own line between the
multi-problem launch and the lane-group coder, which moves with the number of
groups: codes equal to those of separate calls, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth

pytestmark = pytest.mark.gpu
SHAPES = {8: (16, 4), 12: (24, 6), 16: (32, 8)}


@pytest.mark.parametrize("ps,N", [((16,), 7_812), ((16,), 7_813), ((8, 12, 16), 17_240), ((8, 12, 16), 17_250),
                                  ((16,) * 8, 8_000), ((16,) * 8, 16_930)])
@pytest.mark.parametrize("eps", [9.0, 16.0])
def test_batches_equal_separate_calls(gpu_ctx, ps, N, eps):
    g = torch.Generator().manual_seed(N)
    specs = []
    for k, p in enumerate(ps):
        n, s = SHAPES[p]
        Y = torch.randn(N, p, p, generator=g) * torch.exp(torch.randn(N, 1, 1, generator=g) - 1.0)
        D1, D2 = synth.init_dictionaries(p, p, n, n, seed=k)
        specs.append(dict(Y=sdl.signals(Y.cuda()), D1=sdl.dictionary(torch.tensor(np.float32(D1)).cuda()),
                          D2=sdl.dictionary(torch.tensor(np.float32(D2)).cuda()), s=s, eps=eps))
    batch = sdl.Batch(gpu_ctx, specs, autotune=False, graph=False)
    batch.sparse_code()
    batch.sparse_code()
    assert gpu_ctx.status() == 0
    for p, spec in zip(ps, batch.groups):
        ref = gpu_ctx.sparse_code(spec["Y"], spec["D1"], spec["D2"], spec["s"], eps=eps)
        for f in ("support", "coef", "nnz", "res_energy"):
            assert torch.equal(getattr(ref, f), getattr(spec["codes"], f))
    batch.close()
