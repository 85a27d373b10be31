"""The lane-group coder (code-only calls with n1 <= 32, n2 <= 128) at the edges of its
tiles: ragged dictionaries in each compiled tile, counts that leave units of a
warp partly empty, sparsities past the unrolled Cholesky rows, signals so large
that a CTA holds fewer warps, error-driven calls (scan and list), and signals
that are not 16-byte aligned.  Judged by the FP64 oracle within the parity
harness's tolerances."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_03800_gb300 import synth
from parity import check_codes, to_gpu_problem

pytestmark = pytest.mark.gpu

SHAPES = [  # p1, p2, n1, n2, s, N
    (4, 4, 4, 4, 1, 1),
    (7, 9, 13, 15, 5, 129),      # 16 x 16 pairs
    (8, 12, 16, 24, 4, 66),      # 16 x 24
    (9, 8, 17, 16, 4, 31),       # 24 x 16
    (10, 9, 20, 18, 5, 101),     # 20 x 24
    (11, 12, 23, 24, 6, 65),     # 24 x 24
    (8, 16, 15, 31, 6, 70),      # 16 x 32
    (16, 8, 32, 16, 6, 70),      # 32 x 16
    (12, 16, 24, 32, 7, 50),     # 24 x 32
    (16, 12, 31, 23, 8, 50),     # 32 x 24
    (16, 16, 30, 32, 9, 41),     # 32 x 32, first Cholesky row past the unrolled ones
    (8, 8, 16, 16, 12, 40),
    (32, 32, 16, 16, 4, 23),     # 1024-entry signals
    (2, 64, 5, 27, 3, 30),       # the longest side
    (8, 16, 16, 40, 4, 61),      # 16 x 64 pairs: 16 lanes
    (16, 24, 31, 64, 6, 45),     # 32 x 64: one warp per signal
    (9, 30, 15, 100, 5, 40),     # 16 x 128
    (12, 40, 25, 97, 12, 37),    # 32 x 128: teams of two warps, tensor memory, past the unrolled rows
    (16, 64, 32, 128, 10, 331),  # the same with its sizes fixed
    (16, 64, 32, 128, 1, 1),
]


@pytest.mark.parametrize("p1,p2,n1,n2,s,N", SHAPES)
@pytest.mark.parametrize("error_driven", [False, True])
def test_tiles_match_oracle(gpu_ctx, p1, p2, n1, n2, s, N, error_driven):
    rng = np.random.default_rng(500 + 7 * p1 + n2)
    Y = rng.standard_normal((N, p1, p2))
    eps = None
    if error_driven:   # about 40 % start within the target, the others stop before or at s picks
        Y[rng.random(N) < 0.4] *= 0.5
        eps = 0.8 * np.sqrt(p1 * p2)
    D1, D2 = synth.init_dictionaries(p1, p2, n1, n2, seed=2)
    ref = oracle.omp2d(Y, D1, D2, s, eps=eps)
    Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
    got = gpu_ctx.sparse_code(Yg, D1g, D2g, s, eps=eps or 0.0)
    assert gpu_ctx.status() == 0
    check_codes(Y, D1, D2, s, got.support.cpu().numpy(), got.nnz.cpu().numpy(), got.coef.cpu().numpy(),
                got.res_energy.cpu().numpy(), eps=eps, ref=ref).assert_ok()
    # the same signals one float off a 16-byte boundary: the same codes
    flat = torch.empty(Yg.numel() + 1, dtype=torch.float32, device="cuda:0")
    Yv = flat[1:].view(N, p2, p1).transpose(1, 2)
    Yv.copy_(Yg)
    off = gpu_ctx.sparse_code(Yv, D1g, D2g, s, eps=eps or 0.0)
    assert gpu_ctx.status() == 0
    for x, y in zip((got.support, got.coef, got.nnz, got.res_energy),
                    (off.support, off.coef, off.nnz, off.res_energy)):
        assert torch.equal(x, y)


@pytest.mark.parametrize("p,n,s", [(8, 16, 4), (12, 24, 6), (16, 32, 8), (9, 15, 4)])
@pytest.mark.parametrize("eps", [0.0, 5.0])
def test_non_finite_signals_are_reported_alone(gpu_ctx, p, n, s, eps):
    """A NaN and an infinite signal among others get empty codes, NaN energy and
    the error word; their neighbours in the warp keep their codes."""
    rng = np.random.default_rng(9)
    Y = rng.standard_normal((75, p, p))
    D1, D2 = synth.init_dictionaries(p, p, n, n, seed=2)
    Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
    good = gpu_ctx.sparse_code(Yg, D1g, D2g, s, eps=eps)
    assert gpu_ctx.status() == 0
    Yb = Yg.clone()
    Yb[13, 1, 2], Yb[40, 0, 0] = float("nan"), float("inf")
    bad = gpu_ctx.sparse_code(Yb, D1g, D2g, s, eps=eps)
    assert gpu_ctx.status() == -3
    rest = torch.ones(75, dtype=torch.bool, device="cuda:0")
    for k in (13, 40):
        rest[k] = False
        assert bad.nnz[k] == 0 and (bad.support[k] == -1).all() and torch.isnan(bad.res_energy[k])
    assert torch.equal(good.support[rest], bad.support[rest]) and torch.equal(good.coef[rest], bad.coef[rest])
