"""Error-driven coding behind the energy scan: the lines past which a call is scanned,
the number of signals per warp, lists that take several segments of the scratch (and
more than it has), signals that are not finite, and a captured call replayed.  Judged
bit for bit by the same signals coded in calls too small to be scanned."""
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth

pytestmark = pytest.mark.gpu
FIELDS = ("support", "coef", "nnz", "res_energy")


def problem(N, p1, p2, n1, n2, seed):
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    Y = torch.randn(N, p1, p2, device="cuda:0", generator=g)
    Y *= torch.exp(0.5 * torch.randn(N, 1, 1, device="cuda:0", generator=g))
    Y[::97] = 0.0
    D1, D2 = (sdl.dictionary(torch.tensor(D, dtype=torch.float32, device="cuda:0"))
              for D in synth.init_dictionaries(p1, p2, n1, n2, seed=1))
    return sdl.signals(Y), D1, D2


def in_small_calls(ctx, Y, D1, D2, s, eps, step=2000):
    out = sdl.Codes.empty(Y.shape[0], s, Y.device, with_energy=True)
    for k in range(0, Y.shape[0], step):
        c = ctx.sparse_code(Y[k:k + step], D1, D2, s, eps=eps)
        for f in FIELDS:
            getattr(out, f)[k:k + step] = getattr(c, f)
    return out


def same(a, b):
    for f in FIELDS:
        x, y = getattr(a, f), getattr(b, f)
        assert torch.equal(torch.isnan(x.float()), torch.isnan(y.float())), f
        assert torch.equal(torch.nan_to_num(x.float()), torch.nan_to_num(y.float())) and x.dtype == y.dtype, f


@pytest.mark.parametrize("p1,p2,n1,n2,s,N", [
    (8, 8, 16, 16, 4, 32_768), (8, 8, 16, 16, 4, 32_769),      # the line in signals
    (8, 8, 16, 16, 4, 38_913), (8, 8, 16, 16, 4, 77_825), (8, 8, 16, 16, 4, 155_649),   # signals per warp
    (32, 32, 20, 32, 3, 2_048), (32, 32, 20, 32, 3, 2_049), (32, 32, 20, 32, 3, 6_001),  # the line in values
    (9, 7, 13, 15, 5, 33_300), (12, 12, 24, 24, 6, 40_001), (16, 16, 32, 32, 8, 8_193),
])
def test_scanned_calls_equal_small_ones(gpu_ctx, p1, p2, n1, n2, s, N):
    Y, D1, D2 = problem(N, p1, p2, n1, n2, N)
    Y[5, 0, 0], Y[N - 1, 0, 0] = float("nan"), float("inf")
    eps = 0.9 * (p1 * p2) ** 0.5
    got = gpu_ctx.sparse_code(Y, D1, D2, s, eps=eps)
    assert gpu_ctx.status() == -3
    assert got.nnz[5] == 0 and got.nnz[N - 1] == 0
    assert 0.2 < (got.nnz == 0).float().mean().item() < 0.8     # both kinds of signal
    ref = in_small_calls(gpu_ctx, Y, D1, D2, s, eps)
    assert gpu_ctx.status() == -3
    same(got, ref)


def test_lists_of_several_segments():
    p, n, s = 2, 2, 2
    ctx = sdl.Context(0)
    try:
        # a fresh context's scratch: 8 slots per SM of n n + p n floats, less the 4 that hold the count
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        cap = 8 * sms * (n * n + p * n) - 4
        Y, D1, D2 = problem(8 * cap + 1, p, p, n, n, 11)
        eps = 1.8
        ref = in_small_calls(ctx, Y, D1, D2, s, eps, step=30_000)
        for N in (4 * cap - 1, 4 * cap, 4 * cap + 1, 5 * cap + 3, 8 * cap, 8 * cap + 1):
            got = ctx.sparse_code(Y[:N], D1, D2, s, eps=eps)
            assert ctx.status() == 0
            same(got, sdl.Codes(*(getattr(ref, f)[:N] for f in FIELDS)))
    finally:
        ctx.close()


def test_captured_scan_replays(gpu_ctx):
    Y, D1, D2 = problem(50_000, 8, 8, 16, 16, 4)
    out = sdl.Codes.empty(50_000, 4, "cuda:0", with_energy=True)
    ref = gpu_ctx.sparse_code(Y, D1, D2, 4, eps=7.0)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        gpu_ctx.sparse_code(Y, D1, D2, 4, eps=7.0, out=out)
    for _ in range(3):
        for f in FIELDS:
            getattr(out, f).fill_(7)
        graph.replay()
        same(out, ref)
    assert gpu_ctx.status() == 0


def test_first_scan_of_a_context_on_another_stream():
    """The counter is cleared before the context is handed out, also for a stream that
    does not wait for the default one."""
    Y, D1, D2 = problem(40_000, 8, 8, 16, 16, 4)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    ref = None
    for _ in range(8):
        ctx = sdl.Context(0)
        with torch.cuda.stream(side):
            got = ctx.sparse_code(Y, D1, D2, 4, eps=7.0, stream=side)
        assert ctx.status(side) == 0
        ref = ref or got
        same(got, ref)
        ctx.close()
