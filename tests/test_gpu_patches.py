"""Patch extraction and averaging at the edges of their tilings: patch sizes on
both sides of each register tile and past the last one, image widths that are
not multiples of the 32-column or 64-patch runs, one-patch images, the largest
sparsity, and codes without any pick.  Judged by float64 numpy."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth

pytestmark = pytest.mark.gpu

CASES = [  # H, W, p, n, s
    (5, 5, 5, 7, 3),        # one patch
    (40, 33, 1, 2, 1),
    (37, 70, 5, 9, 4),      # patches not a multiple of 16 bytes
    (64, 95, 8, 16, 4),
    (50, 101, 9, 16, 5),
    (71, 140, 12, 24, 6),
    (60, 77, 16, 32, 32),   # the pick list is drained several times
    (45, 90, 17, 20, 8),
    (70, 66, 32, 40, 3),
    (70, 66, 33, 40, 3),    # past the register tiles
    (60, 60, 12, 700, 2),   # dictionaries past the shared-memory staging
]


@pytest.mark.parametrize("H,W,p,n,s", CASES)
def test_patches_and_average_match_numpy(gpu_ctx, H, W, p, n, s):
    rng = np.random.default_rng(H * W + p)
    img = rng.uniform(0, 255, (H, W)).astype(np.float32)
    P, M = synth.all_patches(img.astype(np.float64), p)
    pg, mg = sdl.extract_patches(torch.tensor(img, device="cuda:0"), p)
    # a mean of p^2 values below 256 and one subtraction, in FP32
    tol = 2.0 ** -24 * 256 * (p * p / 32 + 16)
    assert np.abs(mg.cpu().numpy() - M).max() <= tol
    assert np.abs(pg.cpu().numpy() - P).max() <= tol + 2.0 ** -23 * 256

    N = P.shape[0]
    D1, D2 = synth.init_dictionaries(p, p, n, n, seed=4)
    D1, D2 = D1.astype(np.float32), D2.astype(np.float32)
    q = rng.integers(0, n * n, (N, s))
    on = np.arange(s)[None, :] < rng.integers(0, s + 1, N)[:, None]
    x = np.where(on, rng.normal(0, 20, (N, s)), 0.0).astype(np.float32)
    q = np.where(on, q, -1)
    rec = np.einsum("ks,aks,bks->kab", x.astype(np.float64), D1.astype(np.float64)[:, q % n],
                    D2.astype(np.float64)[:, np.maximum(q, 0) // n]) + M[:, None, None]
    acc, cnt = np.zeros((H, W)), np.zeros((H, W))
    rec = rec.reshape(H - p + 1, W - p + 1, p, p)
    for a in range(p):
        for b in range(p):
            acc[a:a + H - p + 1, b:b + W - p + 1] += rec[:, :, a, b]
            cnt[a:a + H - p + 1, b:b + W - p + 1] += 1
    want = acc / cnt
    dev = lambda v, t: torch.tensor(v, dtype=t, device="cuda:0")  # noqa: E731
    codes = sdl.Codes(dev(q, torch.int32), dev(x, torch.float32), dev(on.sum(1), torch.int32))
    got = sdl.patch_average(gpu_ctx, codes, dev(M, torch.float32), sdl.dictionary(dev(D1, torch.float32)),
                            sdl.dictionary(dev(D2, torch.float32)), p, H, W)
    assert gpu_ctx.status() == 0
    # sums of at most p^2 (1 + s) FP32 terms, each below 256 + 80 in size
    assert np.abs(got.cpu().numpy() - want).max() <= 2.0 ** -24 * 336 * (p * (s + 1) + 8)
    none = sdl.Codes(dev(np.full((N, s), -1), torch.int32), dev(np.zeros((N, s)), torch.float32),
                     dev(np.zeros(N), torch.int32))
    flat = sdl.patch_average(gpu_ctx, none, torch.full((N,), 3.0, device="cuda:0"),
                             sdl.dictionary(dev(D1, torch.float32)), sdl.dictionary(dev(D2, torch.float32)), p, H, W)
    assert torch.equal(flat, torch.full_like(flat, 3.0))
