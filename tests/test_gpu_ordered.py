"""A learning pass as coder plus ordered sums must equal the fused pass bit for
bit: the dictionaries of one iteration with the default path against the same with
the shape's first tiling pinned (the fused kernel), at counts around the choice's
line and that leave warps and CTAs unevenly loaded, with a non-finite signal among
them, and against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_03800_gb300 import sdl, synth
from parity import check_iteration, to_gpu_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,s,N", [(8, 16, 4, 8203), (8, 16, 4, 30011), (12, 24, 6, 3647), (12, 24, 6, 20001),
                                     (16, 32, 8, 2051), (16, 32, 8, 9001)])
@pytest.mark.parametrize("bad", [False, True])
def test_iteration_equals_the_fused_pass(gpu_ctx, p, n, s, N, bad):
    imgs = np.stack([synth.synthetic_image(300 + i) for i in range(2)])
    Y = synth.random_patches(imgs, N, p, seed=5)
    Y[::97] = 0.0                                     # codes without picks
    if bad:
        Y[123, 0, 1] = np.nan
    D1, D2 = synth.init_dictionaries(p, p, n, n, seed=1)
    out = []
    try:
        for tiling in (-1, sdl.tilings(p, p, n, n, s)[0]):
            gpu_ctx.set_tiling(p, p, n, n, s, tiling, 0)
            Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
            rmse = torch.zeros(2, dtype=torch.float64, device="cuda:0")
            c = gpu_ctx.iterate(Yg, D1g, D2g, s, rmse_out=rmse)
            assert gpu_ctx.status() == (-3 if bad else 0)
            out.append((D1g, D2g, c.support, c.coef, c.nnz, rmse))
    finally:
        gpu_ctx.set_tiling(p, p, n, n, s, -1)
    for x, y in zip(out[0][:-1], out[1][:-1]):
        assert torch.equal(x, y)
    # the energies are added in another order: FP32 terms, compensated or in FP64
    assert torch.allclose(out[0][-1], out[1][-1], rtol=1e-6, atol=0.0)
    if not bad and N < 4000:
        D1g, D2g, sup, coef, nnz, rmse = (v.cpu().numpy() for v in out[0])
        check_iteration(Y, D1, D2, s, sup, nnz, coef, D1g, D2g, rmse, ref=oracle.iterate(Y, D1, D2, s))
