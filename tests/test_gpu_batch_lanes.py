"""Code-only batches on both sides of the rule that takes them from the
multi-problem launch to the lane-group coder: the codes equal those of the pinned
fused tilings bit for bit, error-driven and not, with zero signals, replayed."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth

pytestmark = pytest.mark.gpu
# p, n, s, a compiled tiling; 256, 576 and 1024 atom pairs
SHAPES = {8: (16, 4, 0), 12: (24, 6, 2), 16: (32, 8, 4)}


@pytest.mark.parametrize("ps,N", [((8, 12, 16), 12_900), ((8, 12, 16), 13_000), ((16,), 7_812), ((16,), 7_813),
                                  ((8, 12), 96_150), ((8, 12), 96_160), ((12,), 1)])
@pytest.mark.parametrize("eps", [0.0, 6.0])
def test_codes_equal_the_pinned_tilings(gpu_ctx, ps, N, eps):
    g = torch.Generator().manual_seed(N)
    specs = []
    for p in ps:
        n, s, _ = SHAPES[p]
        Y = torch.randn(N, p, p, generator=g) * torch.exp(torch.randn(N, 1, 1, generator=g) - 1.0)
        Y[::97] = 0.0
        D1, D2 = synth.init_dictionaries(p, p, n, n, seed=p)
        specs.append(dict(Y=sdl.signals(Y.cuda()), D1=sdl.dictionary(torch.tensor(np.float32(D1)).cuda()),
                          D2=sdl.dictionary(torch.tensor(np.float32(D2)).cuda()), s=s, eps=eps))
    batch = sdl.Batch(gpu_ctx, specs, autotune=False, graph=True)
    batch.sparse_code()
    batch.sparse_code()
    assert gpu_ctx.status() == 0
    for p, spec in zip(ps, batch.groups):
        n, s, tiling = SHAPES[p]
        gpu_ctx.set_tiling(p, p, n, n, s, tiling)
        ref = gpu_ctx.sparse_code(spec["Y"], spec["D1"], spec["D2"], s, eps=eps)
        gpu_ctx.set_tiling(p, p, n, n, s, -1)
        codes = spec["codes"]
        assert torch.equal(ref.nnz, codes.nnz) and torch.equal(ref.support, codes.support)
        assert torch.equal(ref.coef, codes.coef)
