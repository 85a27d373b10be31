"""Sparsities past the unrolled Cholesky rows of the lane-group coder, up to the
largest (32): 8, 16 and 32 lanes and teams of two warps share the rows of the factor.
Counts that leave lanes of a warp without a signal; signals that stop early beside
others that go on.  Judged by the FP64 oracle within the parity harness's tolerances."""
import numpy as np
import pytest

import oracle
from paper_2007_03800_gb300 import synth
from parity import check_codes, to_gpu_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p1,p2,n1,n2", [
    (8, 8, 13, 16),      # 8 lanes
    (12, 12, 24, 24),
    (10, 9, 20, 18),
    (8, 8, 16, 32),
    (16, 12, 30, 32),    # 16 lanes
    (6, 12, 16, 40),
    (8, 16, 32, 64),     # one warp
    (9, 16, 15, 100),
    (8, 24, 31, 97),     # two warps
])
@pytest.mark.parametrize("s", [9, 16, 17, 25, 32])
def test_many_picks_match_oracle(gpu_ctx, p1, p2, n1, n2, s):
    N = 37
    rng = np.random.default_rng(100 * s + n2)
    Y = rng.standard_normal((N, p1, p2))
    D1, D2 = synth.init_dictionaries(p1, p2, n1, n2, seed=2)
    Y[rng.random(N) < 0.4] *= 0.5
    eps = 0.45 * np.sqrt(p1 * p2)   # the halved signals stop after a few picks, the others later
    for e in (None, eps):
        ref = oracle.omp2d(Y, D1, D2, s, eps=e)
        Yg, D1g, D2g = to_gpu_problem(Y, D1, D2)
        got = gpu_ctx.sparse_code(Yg, D1g, D2g, s, eps=e or 0.0)
        assert gpu_ctx.status() == 0
        check_codes(Y, D1, D2, s, got.support.cpu().numpy(), got.nnz.cpu().numpy(), got.coef.cpu().numpy(),
                    got.res_energy.cpu().numpy(), eps=e, ref=ref).assert_ok()
