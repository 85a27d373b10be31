"""The same update check where the other dictionary is wide (its Gram matrix is formed
by each CTA from rows of an odd number of 16-byte pieces: 32, 48 and 64 rows) and on
both sides of the sizes at which the residual energy takes 2 and 4 entries at a time."""
import pytest

import test_gpu_accum

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p1,p2,n1,n2,s,N", [
    (8, 32, 16, 64, 8, 1500),
    (9, 48, 15, 96, 6, 2000),     # 432 entries, rows not a multiple of the lanes
    (16, 64, 32, 128, 10, 3000),  # 1024 entries
    (13, 5, 24, 9, 4, 900),       # 65 entries
    (8, 8, 9, 16, 4, 900),        # 64
    (16, 31, 20, 30, 6, 2000),    # 496
    (19, 27, 30, 32, 6, 2000),    # 513
    (32, 32, 32, 32, 8, 2500),
])
@pytest.mark.parametrize("side", [1, 2])
def test_wide_updates_match_float64(gpu_ctx, p1, p2, n1, n2, s, N, side):
    test_gpu_accum.test_update_matches_float64(gpu_ctx, p1, p2, n1, n2, s, N, side)
