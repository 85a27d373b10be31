"""Input rows of the support network: the 16-byte form against the general one (the same
signals at an address that is not 16-byte aligned give the same bits), at ragged
signal counts and at sizes around the 32-element step."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p1,p2,N", [(2, 2, 1), (8, 8, 33), (4, 9, 131), (6, 10, 64), (12, 12, 515), (3, 5, 70)])
def test_scores_do_not_depend_on_alignment(gpu_ctx, p1, p2, N):
    rng = np.random.default_rng(p1 * p2 + N)
    P, H, n1, n2 = p1 * p2, 40, 4, 6
    net = sdl.MLP(gpu_ctx, p1, p2, n1, n2, hidden=H, max_batch=64)
    W1, W2 = rng.standard_normal((H, P)) * 0.3, rng.standard_normal((n1 * n2, H)) * 0.2
    net.set_weights(W1, np.zeros(H), W2, np.zeros(n1 * n2))
    buf = torch.zeros(N * P + 4, device="cuda:0")
    sig = torch.tensor(rng.standard_normal(N * P), dtype=torch.float32, device="cuda:0")
    sig[:P] = 0.0                                   # a zero signal: zero row
    outs = []
    for off in (0, 1, 2):
        buf[off:off + N * P] = sig
        outs.append(net.forward(buf[off:off + N * P].view(N, p2, p1).transpose(1, 2)).cpu())
    assert gpu_ctx.status() == 0
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    x = sig.view(N, P).double().cpu()
    x = x / x.norm(dim=1, keepdim=True).clamp_min(1e-30)
    h = torch.nn.functional.gelu(x @ torch.tensor(W1).T)
    ref = h @ torch.tensor(W2).T
    assert (outs[0].double() - ref).norm() <= 2.0 ** -6 * ref.norm()
    net.close()
