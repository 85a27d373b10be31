"""The shortlist coder at ragged calls: one signal, counts that are no multiple of a
warp's signals, short and full lists, lists in rows longer than the part that is
used, empty lists, zero and non-finite signals, unaligned signals."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth
from parity import to_gpu_problem

pytestmark = pytest.mark.gpu
SHAPES = {8: (16, 4), 12: (24, 6)}


def problem(p, N, k2, seed):
    n, s = SHAPES[p]
    Y, D1, D2, _, _ = synth.kron_model(N, p, p, n, n, s, 15.0, seed=seed)
    rng = np.random.default_rng(seed)
    cand = np.stack([rng.permutation(n * n)[:k2] for _ in range(N)]).astype(np.int32)
    return Y, D1, D2, s, cand


@pytest.mark.parametrize("p", [8, 12])
@pytest.mark.parametrize("N,k1,k2", [(1, 32, 32), (3, 1, 1), (131, 5, 9), (2050, 32, 48), (1024, 31, 31)])
def test_codes_and_flags_match_the_oracle(gpu_ctx, p, N, k1, k2):
    Y, D1, D2, s, cand = problem(p, N, k2, 5 + N + k1)
    if N > 100:
        cand[7, :] = -1                # nothing to pick
        cand[11, 1:] = -1              # one pair only
        Y[13] = 0.0
    Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
    cg = torch.tensor(cand, device="cuda:0")
    codes, flag = gpu_ctx.sparse_code_shortlist(Yg, D1g, D2g, s, cg, k1)
    assert gpu_ctx.status() == 0
    sup, nnz = codes.support.cpu().numpy(), codes.nnz.cpu().numpy()
    coef, e = codes.coef.cpu().numpy(), codes.res_energy.cpu().numpy()
    Q = D1.shape[1] * D2.shape[1]
    for k in range(N):
        allowed = set(int(q) for q in cand[k, :k1] if q >= 0)
        got = sup[k, :nnz[k]]
        assert set(got) <= allowed and len(set(got)) == nnz[k] and np.all(sup[k, nnz[k]:] == -1)
        if not Y[k].any():
            assert nnz[k] == 0 and flag[k].item() == 0
            continue
        assert nnz[k] == min(s, len(allowed))
        # least squares on the picks, and greedy picks by replay (ties within rounding)
        A = np.stack([np.outer(D1[:, q % D1.shape[1]], D2[:, q // D1.shape[1]]).ravel() for q in got], 1) \
            if nnz[k] else np.zeros((p * p, 0))
        y = Y[k].ravel()
        weakest = np.inf
        for t in range(nnz[k]):
            x = np.linalg.lstsq(A[:, :t], y, rcond=None)[0] if t else np.zeros(0)
            c = np.abs(np.einsum("ai,ab,bj->ji", D1, (y - A[:, :t] @ x).reshape(p, p), D2).ravel())
            best = max(c[q] for q in allowed - set(got[:t]))
            assert c[got[t]] >= best - 1e-4 * np.linalg.norm(y)
            weakest = min(weakest, c[got[t]])
        if nnz[k]:
            x = np.linalg.lstsq(A, y, rcond=None)[0]
            tol = np.linalg.cond(A) ** 2 * 2.0 ** -24 * 64
            assert np.linalg.norm(coef[k, :nnz[k]] - x) <= tol * np.linalg.norm(x)
            r = y - A @ x
            assert abs(e[k] - r @ r) <= 1e-5 * (y @ y)
            c = np.abs(np.einsum("ai,ab,bj->ji", D1, r.reshape(p, p), D2).ravel())
            rest = max(c[q] for q in range(Q) if q not in set(got))
            if nnz[k] < s:
                assert flag[k].item() == 0
            elif abs(rest - 0.7 * weakest) > 1e-4 * np.linalg.norm(y):
                assert flag[k].item() == int(rest > 0.7 * weakest)


@pytest.mark.parametrize("p", [8, 12])
def test_alignment_and_non_finite_signals(gpu_ctx, p):
    N = 203
    Y, D1, D2, s, cand = problem(p, N, 32, 3)
    Y[5, 1, 2] = np.inf
    Y[6, 0, 0] = np.nan
    Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
    cg = torch.tensor(cand, device="cuda:0")
    a, fa = gpu_ctx.sparse_code_shortlist(Yg, D1g, D2g, s, cg, 32)
    buf = torch.zeros(N * p * p + 1, device="cuda:0")
    buf[1:] = Yg.transpose(1, 2).reshape(-1)
    b, fb = gpu_ctx.sparse_code_shortlist(buf[1:].view(N, p, p).transpose(1, 2), D1g, D2g, s, cg, 32)
    assert gpu_ctx.status() == 0
    for k in (5, 6):
        assert fa[k].item() == 1 and a.nnz[k].item() == 0
    assert torch.equal(fa, fb) and torch.equal(a.support, b.support) and torch.equal(a.coef, b.coef)
