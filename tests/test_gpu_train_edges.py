"""Training kernels and the long-K GEMM at ragged sizes: batches and layers that
are not multiples of the 32-signal, 64-score and 32 x 32 blocks, and GEMMs whose
few output tiles take the narrow 128 x 32 form."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2007_03800_gb300 import sdl, synth
from parity import to_gpu_problem

pytestmark = pytest.mark.gpu


def bf16(a):
    return torch.tensor(np.asarray(a, dtype=np.float32)).to(torch.bfloat16).double().numpy()


@pytest.mark.parametrize("p1,p2,n1,n2,H,B,s", [(8, 8, 16, 16, 40, 72, 4), (6, 7, 10, 12, 72, 40, 3), (4, 4, 2, 4, 8, 8, 1),
                                               (12, 12, 24, 24, 136, 1032, 6)])
def test_gradients_at_ragged_sizes(gpu_ctx, p1, p2, n1, n2, H, B, s):
    rng = np.random.default_rng(B + H)
    Q, P = n1 * n2, p1 * p2
    Y = rng.standard_normal((B, p1, p2))
    labels = np.array([rng.choice(Q, s, replace=False) for _ in range(B)])
    labels[rng.random(labels.shape) < 0.1] = -1        # unused slots
    W1, b1 = rng.standard_normal((H, P)) * 0.2, rng.standard_normal(H) * 0.1
    W2, b2 = rng.standard_normal((Q, H)) * 0.2, rng.standard_normal(Q) * 0.1
    net = sdl.MLP(gpu_ctx, p1, p2, n1, n2, hidden=H, max_batch=B + 8)
    net.set_weights(W1, b1, W2, b2)
    D1, D2 = synth.init_dictionaries(p1, p2, n1, n2)
    Yg, _, _ = to_gpu_problem(Y, D1, D2)
    sup = torch.tensor(labels, dtype=torch.int32, device="cuda:0")
    loss, g = net.gradients(Yg, sup)
    assert gpu_ctx.status() == 0
    T = np.zeros((B, Q))
    for k in range(B):
        T[k, labels[k][labels[k] >= 0]] = 1.0
    ref_loss, ref = omlp.loss_and_grads(bf16(omlp.inputs(Y)), T, bf16(W1), b1, bf16(W2), b2)
    assert abs(loss - ref_loss) / ref_loss < 1e-2
    for name in ("W1", "b1", "W2", "b2"):
        err = np.linalg.norm(g[name] - ref[name]) / np.linalg.norm(ref[name])
        assert err < 3e-2, (name, err)
    # a step with these gradients moves every weight by lr against the sign of
    # its gradient (first Adam step), where that is far from zero
    net.train_step(Yg, sup, 1e-3)
    assert gpu_ctx.status() == 0
    for name, w0, w in zip(("W1", "b1", "W2", "b2"), (W1, b1, W2, b2), net.get_weights()):
        big = np.abs(g[name]) > 1e-5
        moved = (w - w0.astype(np.float32)) * np.sign(g[name])
        assert np.all(np.abs(moved[big] + 1e-3) < 2e-5), name
    net.close()


@pytest.mark.parametrize("M,N,K", [(512, 152, 4096), (100, 33, 1024), (1000, 8, 1088), (1, 1, 1500), (300, 40, 2056)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_long_k_gemm_matches_float64(gpu_ctx, M, N, K, accumulate):
    g = torch.Generator().manual_seed(M + N)
    ld = (K + 7) // 8 * 8
    A = torch.randn(M, ld, generator=g).to(torch.bfloat16)
    B = torch.randn(N, ld, generator=g).to(torch.bfloat16)
    C0 = torch.randn(M, N, generator=g)
    A, B, C = A.cuda()[:, :K], B.cuda()[:, :K], C0.cuda()
    sdl.gemm_bf16(gpu_ctx, A, B, alpha=0.5, C=C, accumulate=accumulate)
    assert gpu_ctx.status() == 0
    a, b = A.double().cpu(), B.double().cpu()
    want = 0.5 * (a @ b.t()) + (C0.double() if accumulate else 0.0)
    # K FP32 additions of exact products, relative to the sum of their sizes
    bound = K * 2.0 ** -23 * (a.abs() @ b.abs().t()) + 2.0 ** -22 * want.abs()
    assert bool(((C.double().cpu() - want).abs() <= bound).all())
