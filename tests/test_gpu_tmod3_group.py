"""Two signals per warp in the three-mode coder: counts that leave a unit half
empty, and signals without a code (zero, non-finite) beside others.  A signal's
code does not depend on its neighbours."""
import numpy as np
import pytest
import torch

from oracle import tmod3
from paper_2007_03800_gb300 import sdl, synth
from parity import check_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,s", [((4, 4, 4), (8, 8, 8), 4), ((4, 4, 16), (8, 8, 16), 8)])
@pytest.mark.parametrize("N", [1, 2, 77])
def test_counts_and_empty_signals(gpu_ctx, p, n, s, N):
    Y, _, _, _ = synth.kron_model3(N, p, n, s, 20.0, seed=82)
    rng = np.random.default_rng(2)
    Ds = [synth.random_dictionary(p[m], n[m], rng) for m in range(3)]
    Dg = [sdl.dictionary(torch.tensor(D, dtype=torch.float32, device="cuda:0")) for D in Ds]

    def code(A):
        out = gpu_ctx.sparse_code3(sdl.signals3(torch.tensor(A, dtype=torch.float32, device="cuda:0")), *Dg, s)
        return gpu_ctx.status(), out

    st, out = code(Y)
    assert st == 0
    check_codes(Y, None, None, s, out.support.cpu().numpy(), out.nnz.cpu().numpy(), out.coef.cpu().numpy(),
                ref=tmod3.omp3d(Y, *Ds, s),
                replay=lambda Yo, so, no: tmod3.omp3d_replay(Yo, *Ds, so, no, s)).assert_ok()
    if N < 8:
        return
    B = Y.copy()
    B[4] = 0.0
    B[7, 0, 1, 2] = np.nan
    st, bad = code(B)
    assert st == -3
    rest = torch.ones(N, dtype=torch.bool, device="cuda:0")
    rest[[4, 7]] = False
    for k in (4, 7):
        assert bad.nnz[k] == 0 and (bad.support[k] == -1).all() and (bad.coef[k] == 0).all()
    assert bad.res_energy[4] == 0 and torch.isnan(bad.res_energy[7])
    assert torch.equal(out.support[rest], bad.support[rest]) and torch.equal(out.coef[rest], bad.coef[rest])
