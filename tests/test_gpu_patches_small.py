"""Patch averaging on both sides of the line at which a small image with many slots is
rebuilt from written patches."""
import pytest

import test_gpu_patches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,p,n,s", [
    (50, 50, 8, 16, 5), (50, 50, 8, 16, 6),       # the line lies between
    (50, 50, 8, 16, 32), (40, 700, 8, 16, 31), (40, 700, 8, 16, 32),
    (80, 81, 16, 32, 15), (80, 81, 16, 32, 16), (31, 30, 6, 11, 9), (24, 50, 24, 30, 32),
])
def test_small_images_match_numpy(gpu_ctx, H, W, p, n, s):
    test_gpu_patches.test_patches_and_average_match_numpy(gpu_ctx, H, W, p, n, s)
