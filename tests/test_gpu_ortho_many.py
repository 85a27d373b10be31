"""Orthonormal codes on both sides of the lines between the lane groups and a warp per
signal (many kept entries, few signals): the same signals give the same codes, and
those are the s largest entries of D1^T Y D2."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p1,p2,s", [(8, 8, 24), (8, 8, 25), (10, 6, 32), (16, 16, 32), (4, 8, 16), (4, 8, 32), (3, 7, 21)])
def test_codes_do_not_depend_on_the_form(gpu_ctx, p1, p2, s):
    rng = np.random.default_rng(p1 + s)
    D1, D2 = (np.linalg.qr(rng.standard_normal((p, p)))[0] for p in (p1, p2))
    Y = rng.standard_normal((50_001, p1, p2)).astype(np.float32)
    Yg = sdl.signals(torch.tensor(Y, device="cuda:0"))
    D1g, D2g = (sdl.dictionary(torch.tensor(D, dtype=torch.float32, device="cuda:0")) for D in (D1, D2))
    full = gpu_ctx.ortho_sparse_code(Yg, D1g, D2g, s)
    assert gpu_ctx.status() == 0
    for N in (50_000, 8193, 8192, 33, 1):
        part = gpu_ctx.ortho_sparse_code(Yg[:N], D1g, D2g, s)
        assert gpu_ctx.status() == 0
        for f in ("support", "coef", "nnz"):
            assert torch.equal(getattr(part, f), getattr(full, f)[:N]), (N, f)
    C = np.einsum("ai,kab,bj->kij", D1.astype(np.float32).astype(np.float64), Y[:200].astype(np.float64),
                  D2.astype(np.float32).astype(np.float64))
    flat = C.transpose(0, 2, 1).reshape(200, -1)                   # q = i + p1 j
    sup, coef = full.support[:200].cpu().numpy(), full.coef[:200].cpu().numpy()
    got = np.take_along_axis(flat, sup.astype(np.int64), 1)
    # an entry is a sum of p1 p2 products of FP32 values, in two stages
    tol = (p1 + p2) * 2.0 ** -24 * np.linalg.norm(flat, axis=1, keepdims=True)
    assert (np.abs(got - coef) <= tol).all()
    want = -np.sort(-np.abs(flat), axis=1)[:, :s]
    assert (np.abs(want - np.abs(got)) <= 2 * tol).all()
