"""Dictionary updates from given codes at the edges of the lane-per-atom partial
sums: row counts on both sides of the register tiles, atoms at and past the lane
limit (the larger side takes the general kernel), contraction lengths that are
not multiples of a chunk, empty and repeated picks, signals off a 16-byte
boundary, and the objective asked for or not.  Judged by a float64 update."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth
from parity import to_gpu_problem

pytestmark = pytest.mark.gpu

SHAPES = [  # p1, p2, n1, n2, s, N
    (8, 8, 16, 16, 4, 700),
    (7, 9, 13, 18, 5, 333),
    (12, 12, 24, 24, 6, 901),
    (16, 16, 32, 32, 8, 1501),
    (17, 5, 32, 7, 3, 800),       # 32-row tile, two chunks on the other side
    (4, 40, 8, 33, 6, 1200),      # 40 rows and 33 atoms: side D2 in the general kernel
    (32, 20, 32, 24, 12, 1500),
    (6, 6, 6, 6, 32, 400),        # most picks repeat an atom
]


def update64(Y, D1, D2, q, x, side):
    n1, n2 = D1.shape[1], D2.shape[1]
    X = np.zeros((Y.shape[0], n1, n2))
    for l in range(q.shape[1]):
        on = q[:, l] >= 0
        np.add.at(X, (np.nonzero(on)[0], q[on, l] % n1, q[on, l] // n1), x[on, l])
    before = ((Y - D1 @ X @ D2.T) ** 2).sum()
    if side == 1:
        T = X @ D2.T
        P, B = np.einsum("kib,kjb->ij", T, T), np.einsum("kab,kib->ai", Y, T)
    else:
        T = D1 @ X
        P, B = np.einsum("kaj,kal->jl", T, T), np.einsum("kab,kaj->bj", Y, T)
    D = np.linalg.solve(P, B.T).T
    after = ((Y - (D @ X @ D2.T if side == 1 else D1 @ X @ D.T)) ** 2).sum()
    norm = np.linalg.norm(D, axis=0)
    return D / norm, norm, before, after, np.linalg.cond(P)


@pytest.mark.parametrize("p1,p2,n1,n2,s,N", SHAPES)
@pytest.mark.parametrize("side", [1, 2])
def test_update_matches_float64(gpu_ctx, p1, p2, n1, n2, s, N, side):
    rng = np.random.default_rng(70 + p1 + 3 * n2)
    D1, D2 = synth.init_dictionaries(p1, p2, n1, n2, seed=3)
    D1, D2 = D1.astype(np.float32).astype(np.float64), D2.astype(np.float32).astype(np.float64)
    q = rng.integers(0, n1 * n2, (N, s))
    q = np.where(rng.random((N, s)) < 0.15, -1, q)            # empty slots anywhere
    x = np.where(rng.random((N, s)) < 0.05, 0.0, rng.standard_normal((N, s))).astype(np.float32)
    Y = np.zeros((N, p1, p2))
    for l in range(s):
        on = (q[:, l] >= 0)[:, None, None]
        Y += on * x[:, l, None, None] * np.einsum("ak,bk->kab", D1[:, q[:, l] % n1], D2[:, np.maximum(q[:, l], 0) // n1])
    Y = (Y + 0.3 * rng.standard_normal(Y.shape)).astype(np.float32).astype(np.float64)
    D, norm, before, after, cond = update64(Y, D1, D2, q, x.astype(np.float64), side)
    want_x = x * norm[(q % n1) if side == 1 else np.maximum(q, 0) // n1]
    want_x = np.where(q >= 0, want_x, x)

    def run(aligned, objective):
        Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
        if not aligned:
            flat = torch.empty(Yg.numel() + 1, dtype=torch.float32, device="cuda:0")
            Yv = flat[1:].view(N, p2, p1).transpose(1, 2)
            Yv.copy_(Yg)
            Yg = Yv
        codes = sdl.Codes(torch.tensor(q, dtype=torch.int32, device="cuda:0"), torch.tensor(x, device="cuda:0"),
                          torch.full((N,), s, dtype=torch.int32, device="cuda:0"))
        obj = torch.zeros(2, dtype=torch.float64, device="cuda:0") if objective else None
        (gpu_ctx.update_D1 if side == 1 else gpu_ctx.update_D2)(Yg, D1g, D2g, codes, objective_out=obj)
        assert gpu_ctx.status() == 0
        return (D1g if side == 1 else D2g).cpu().numpy(), codes.coef.cpu().numpy(), obj

    # the FP32 sums (N terms, compensated in part) through the normal equations
    tol = cond * 2.0 ** -24 * 64
    for aligned in (True, False):
        for objective in (False, True):
            gD, gx, obj = run(aligned, objective)
            assert np.linalg.norm(gD - D) <= tol * np.linalg.norm(D)
            assert np.linalg.norm(gx - want_x) <= tol * np.linalg.norm(want_x)
            if objective:
                o = obj.cpu().numpy()
                assert abs(o[0] - before) <= 1e-5 * before and abs(o[1] - after) <= 1e-5 * before
