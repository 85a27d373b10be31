"""The orthonormal variant through the lane-group coder (fixed sparsity) against
the one-signal-per-warp kernels, which a positive error target that is never
reached still selects: codes bit for bit at every tile, and one learning
iteration bit for bit at the square shapes where coding and sums are split."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl

pytestmark = pytest.mark.gpu

NEVER = 1e-10      # its square is positive, and far below any residual energy here


def problem(p1, p2, N, seed):
    g = torch.Generator().manual_seed(seed)
    Y = torch.randn(N, p1, p2, generator=g)
    Q = [torch.linalg.qr(torch.randn(p, p, generator=g, dtype=torch.float64))[0].float() for p in (p1, p2)]
    return sdl.signals(Y.cuda()), [sdl.dictionary(q.cuda()) for q in Q]


@pytest.mark.parametrize("p1,p2,s,N", [(8, 8, 4, 501), (12, 12, 6, 333), (16, 16, 8, 203), (12, 12, 16, 33),
                                       (16, 16, 20, 35), (7, 9, 5, 130), (1, 3, 2, 9), (16, 11, 8, 67), (20, 31, 6, 41),
                                       (32, 32, 12, 30), (32, 5, 3, 50)])
def test_codes_equal_the_one_warp_kernels(gpu_ctx, p1, p2, s, N):
    Y, (D1, D2) = problem(p1, p2, N, 3)
    a = gpu_ctx.ortho_sparse_code(Y, D1, D2, s)
    b = gpu_ctx.ortho_sparse_code(Y, D1, D2, s, eps=NEVER)
    assert gpu_ctx.status() == 0
    for x, y in zip((a.support, a.coef, a.nnz, a.res_energy), (b.support, b.coef, b.nnz, b.res_energy)):
        assert torch.equal(x, y)


@pytest.mark.parametrize("p,s,N", [(8, 4, 24001), (8, 16, 30007), (12, 6, 11003), (12, 1, 20011), (16, 8, 6007)])
def test_iteration_equals_the_fused_pass(gpu_ctx, p, s, N):
    out = []
    for eps in (0.0, NEVER):
        Y, (D1, D2) = problem(p, p, N, 4)
        Y[::101] = 0.0
        rmse = torch.zeros(2, dtype=torch.float64, device="cuda:0")
        for _ in range(2):
            c = gpu_ctx.ortho_iterate(Y, D1, D2, s, eps=eps, rmse_out=rmse)
        assert gpu_ctx.status() == 0
        out.append((D1, D2, c.support, c.coef, c.nnz, rmse))
    for x, y in zip(out[0][:-1], out[1][:-1]):
        assert torch.equal(x, y)
    assert np.allclose(out[0][-1].cpu(), out[1][-1].cpu(), rtol=1e-6, atol=0.0)
