"""The GEMM on both sides of the lines between its epilogues: contraction lengths per
tile width, accumulations within and past the size at which 16 warps hold up the
reduce-adds, and narrow tiles.  Against an FP64 product of the same BF16 operands, on
rows spread over the output; FP32 accumulation in K / 16 instructions of 16 products
is within K / 16 half ulps of the largest sum."""
import pytest
import torch

from paper_2007_03800_gb300 import sdl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (2000, 576, 768), (2000, 576, 776), (20_000, 1024, 1024), (20_000, 1024, 1032),
    (6144, 4096, 64), (6160, 4096, 64), (43_700, 576, 200),     # 96 MB of FP32 output, just over, and ragged
    (1152, 128, 1016), (1152, 128, 1024), (1153, 128, 1024), (130, 36, 2048),
])
@pytest.mark.parametrize("accumulate", [False, True])
def test_lines_match_fp64(gpu_ctx, M, N, K, accumulate):
    g = torch.Generator(device="cuda:0").manual_seed(M + K)
    A = torch.randn(M, K, device="cuda:0", generator=g).bfloat16()
    B = torch.randn(N, K, device="cuda:0", generator=g).bfloat16()
    C = torch.randn(M, N, device="cuda:0", generator=g)
    rows = torch.unique(torch.cat([torch.arange(0, M, max(1, M // 97), device="cuda:0"),
                                   torch.arange(max(0, M - 5), M, device="cuda:0")]))
    ref = A[rows].double() @ B.double().t() + (C[rows].double() if accumulate else 0.0)
    sdl.gemm_bf16(gpu_ctx, A, B, C=C, accumulate=accumulate)
    assert gpu_ctx.status() == 0
    err = (C[rows].double() - ref).abs().max().item()
    assert err <= (K / 16 + 2) * 2.0 ** -24 * ref.abs().max().item(), err
