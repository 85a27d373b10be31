"""Network calls allocate nothing once the network exists: the first forward pass of a
context over more signals than a training batch, and the first training step, can
be captured into a CUDA graph, and the graph stays valid when later calls grow the
context's workspaces."""
import numpy as np
import pytest
import torch

from paper_2007_03800_gb300 import sdl, synth

pytestmark = pytest.mark.gpu
P, N_ATOMS, S, H = 8, 16, 4, 64


def network(ctx, max_batch=64):
    m = sdl.MLP(ctx, P, P, N_ATOMS, N_ATOMS, hidden=H, max_batch=max_batch)
    m.init(3)
    return m


def capture(fn):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out = fn()
    return graph, out


@pytest.mark.parametrize("N", [64, 65, 1000, 32_768 + 5])
def test_first_forward_can_be_captured(N):
    g = torch.Generator(device="cuda:0").manual_seed(N)
    Y = sdl.signals(torch.randn(N, P, P, device="cuda:0", generator=g))
    D1, D2 = (sdl.dictionary(torch.tensor(D, dtype=torch.float32, device="cuda:0"))
              for D in synth.init_dictionaries(P, P, N_ATOMS, N_ATOMS, seed=1))
    ctx = sdl.Context(0)
    try:
        m = network(ctx)
        graph, out = capture(lambda: m.forward(Y))
        # a larger learned-coder call grows the context's workspace
        big = sdl.signals(torch.randn(2 * N + 50_000, P, P, device="cuda:0", generator=g))
        m.sparse_code(big, D1, D2, S)
        graph.replay()
        ref = m.forward(Y)
        assert ctx.status() == 0
        assert torch.equal(out, ref)
        m.close()
    finally:
        ctx.close()


def test_first_training_step_can_be_captured():
    g = torch.Generator(device="cuda:0").manual_seed(5)
    Y = sdl.signals(torch.randn(64, P, P, device="cuda:0", generator=g))
    lab = torch.randint(0, N_ATOMS * N_ATOMS, (64, S), device="cuda:0", generator=g, dtype=torch.int32)
    weights = []
    for captured in (False, True):
        ctx = sdl.Context(0)
        try:
            m = network(ctx)
            if captured:
                graph, _ = capture(lambda: m.train_step(Y, lab, 1e-3))
                graph.replay()
            else:
                m.train_step(Y, lab, 1e-3)
            assert ctx.status() == 0
            weights.append(m.get_weights())
            m.close()
        finally:
            ctx.close()
    for a, b in zip(*weights):
        assert np.array_equal(a, b)
