"""The n <= 32 dictionary solve at its edges: one atom, the largest n and p, atoms
that no code uses (gathered around), a singular normal matrix and non-finite sums
(dictionary untouched, error reported).  Judged in float64."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth
from parity import to_gpu_problem

pytestmark = pytest.mark.gpu


def run(ctx, Y, D1, D2, q, x):
    Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
    codes = sdl.Codes(torch.tensor(q, dtype=torch.int32, device="cuda:0"),
                      torch.tensor(x, dtype=torch.float32, device="cuda:0"),
                      torch.full((q.shape[0],), q.shape[1], dtype=torch.int32, device="cuda:0"))
    obj = torch.zeros(2, dtype=torch.float64, device="cuda:0")
    ctx.update_D1(Yg, D1g, D2g, codes, objective_out=obj)
    return ctx.status(), D1g.cpu().numpy().astype(np.float64), codes.coef.cpu().numpy(), obj.cpu().numpy()


@pytest.mark.parametrize("p1,p2,n1,n2,used", [(3, 4, 1, 5, 1), (8, 8, 32, 16, 32), (64, 8, 32, 8, 32), (64, 8, 31, 8, 17),
                                              (5, 9, 12, 6, 3), (12, 12, 24, 24, 23)])
def test_used_atoms(gpu_ctx, p1, p2, n1, n2, used):
    rng = np.random.default_rng(p1 + n1)
    D1, D2 = (d.astype(np.float32).astype(np.float64) for d in synth.init_dictionaries(p1, p2, n1, n2, seed=6))
    N, s = 2000, 3
    atoms = np.sort(rng.choice(n1, used, replace=False))
    q = atoms[rng.integers(0, used, (N, s))] + n1 * rng.integers(0, n2, (N, s))
    x = rng.standard_normal((N, s)).astype(np.float32).astype(np.float64)
    Y = np.einsum("ks,aks,bks->kab", x, D1[:, q % n1], D2[:, q // n1])
    Y = (Y + 0.2 * rng.standard_normal(Y.shape)).astype(np.float32).astype(np.float64)
    T = np.zeros((N, n1, p2))
    for l in range(s):
        np.add.at(T, (np.arange(N), q[:, l] % n1), x[:, l, None] * D2[:, q[:, l] // n1].T)
    P, B = np.einsum("kib,kjb->ij", T, T), np.einsum("kab,kib->ai", Y, T)
    u = np.ix_(atoms, atoms)
    Du = np.linalg.solve(P[u], B[:, atoms].T).T
    norm = np.ones(n1)
    norm[atoms] = np.linalg.norm(Du, axis=0)
    want = D1.copy()
    want[:, atoms] = Du / norm[atoms]
    after = ((Y - np.einsum("ai,kib->kab", want * norm, T)) ** 2).sum()
    st, D, coef, obj = run(gpu_ctx, Y, D1, D2, q, x)
    tol = np.linalg.cond(P[u]) * 2.0 ** -24 * 64
    assert st == 0
    assert np.linalg.norm(D - want) <= tol * np.linalg.norm(want)
    assert np.array_equal(np.delete(D, atoms, axis=1), np.delete(D1, atoms, axis=1))
    assert np.linalg.norm(coef - x * norm[q % n1]) <= tol * np.linalg.norm(coef)
    assert abs(obj[1] - after) <= 1e-5 * obj[0]


@pytest.mark.parametrize("kind,code", [("singular", -4), ("nonfinite", -3)])
def test_failed_update_leaves_the_dictionary(gpu_ctx, kind, code):
    rng = np.random.default_rng(3)
    p, n, N = 8, 16, 500
    D1, D2 = (d.astype(np.float32).astype(np.float64) for d in synth.init_dictionaries(p, p, n, n, seed=6))
    q = np.stack([rng.integers(0, n * n, N), np.full(N, 3 + 5 * n), np.full(N, 7 + 5 * n)], axis=1)
    x = rng.standard_normal((N, 3))
    x[:, 2] = x[:, 1]                          # atoms 3 and 7 always together, same weight
    q[:, 0] = np.where(np.isin(q[:, 0] % n, (3, 7)), 0, q[:, 0])
    Y = rng.standard_normal((N, p, p))
    if kind == "nonfinite":
        x[17, 0] = 3e38                        # overflows in the sums
    st, D, coef, _ = run(gpu_ctx, Y, D1, D2, q, x)
    assert st == code
    assert np.array_equal(D, D1) and np.array_equal(coef, x.astype(np.float32))
