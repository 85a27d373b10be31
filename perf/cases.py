"""What the framework is timed on: calls of its public entry points, each at the
sizes of a configuration of this repository or at ragged sizes between them.

  listed()             the named cases (what each stands for is said beside it)
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs on the GPU, made from the seed alone, and the context,
                       batch or network that a program keeps
  run(state)           one pass through the entry points, and its outputs
  work(case)           bytes and operations that one pass cannot do without
  exact(case, seed)    the outputs in 64 bits, by plain torch
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2007_03800_gb300 import learned, sdl

DEV = "cuda:0"

# sizes of the three groups of the mixed denoising workload: p, n, s
GROUPS = {8: (8, 16, 4), 12: (12, 24, 6), 16: (16, 32, 8)}


def listed():
    return [
        # the parity workload: a few thousand 8 x 8 signals, where launches and latency count
        dict(name="code_8x8_4k", kind="code", data="model", N=4096, p1=8, p2=8, n1=16, n2=16, s=4),
        # sparse coding of 12 x 12 image patches with the dictionaries of the patch-learning workload
        dict(name="code_12x12_200k", kind="code", data="patches", N=200000, p1=12, p2=12, n1=24, n2=24, s=6),
        # a user's own sizes: unequal sides, an odd count and sparsity, no size a multiple of another
        dict(name="code_10x9_100k", kind="code", data="model", N=99991, p1=10, p2=9, n1=20, n2=18, s=5),
        # hyperspectral-shaped signals (pixels x bands), wide dictionaries
        dict(name="code_16x64_50k", kind="code", data="hyper", N=50000, p1=16, p2=64, n1=32, n2=128, s=10),
        # the final coding of the denoising pipeline: every patch of three sizes, error-driven, one batch
        dict(name="denoise_code_512", kind="batch", H=512, W=512, sigma=20.0, groups="8,12,16"),
        # gathering an image's patches, and the image put together again from coded patches
        dict(name="denoise_io_512", kind="io", H=512, W=512, p=12, n=24, s=6),
        # one iteration of dictionary learning on image patches (the headline)
        dict(name="learn_12x12_200k", kind="learn", N=200000, p=12, n=24, s=6),
        # the two dictionary updates on their own, with codes in hand (16 x 16 patches)
        dict(name="update_16x16_100k", kind="update", N=100000, p1=16, p2=16, n1=32, n2=32, s=8),
        # one iteration with orthonormal dictionaries on image patches
        dict(name="ortho_12x12_200k", kind="ortho", N=200000, p1=12, p2=12, s=6),
        # three-mode coding of hyperspectral-shaped cubes
        dict(name="code3_4x4x16_50k", kind="code3", N=50000, p1=4, p2=4, p3=16, n1=8, n2=8, n3=16, s=8),
        # an epoch of training of the support-proposal network (forward, backward, Adam)
        dict(name="train_144_512_576", kind="train", N=65536, batch=4096, p=12, n=24, s=6, hidden=512),
        # coding through the proposal network's shortlists, with fallback and guard
        dict(name="learned_8x8_200k", kind="learned", N=200000, p=8, n=16, s=4, k=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["code", "code", "code", "wide", "batch", "io", "learn", "learn", "update", "update",
                       "ortho", "code3", "train", "learned"])
    if kind == "code":
        p1, p2 = rng.randint(6, 16), rng.randint(6, 16)
        n1, n2 = rng.randint(p1, 2 * p1), rng.randint(p2, 2 * p2)
        s = rng.randint(2, 8)
        most = min(250000, int(2.0e9 / (n1 * n2 * s)))
        return dict(kind="code", data=rng.choice(["model", "patches"]), N=_log(rng, 1500, most), p1=p1, p2=p2,
                    n1=n1, n2=n2, s=s)
    if kind == "wide":
        p1, p2 = rng.randint(8, 16), rng.randint(24, 64)
        n1, n2 = rng.randint(p1, 2 * p1), rng.randint(p2, 2 * p2)
        s = rng.randint(4, 10)
        return dict(kind="code", data="hyper", N=_log(rng, 1000, min(60000, int(2.0e9 / (n1 * n2 * s)))), p1=p1,
                    p2=p2, n1=n1, n2=n2, s=s)
    if kind == "batch":
        return dict(kind="batch", H=rng.randint(150, 512), W=rng.randint(150, 512), sigma=float(rng.randint(10, 40)),
                    groups=rng.choice(["8,12", "8,16", "12,16", "8,12,16", "12"]))
    if kind == "io":
        p = rng.randint(6, 16)
        return dict(kind="io", H=rng.randint(120, 640), W=rng.randint(120, 640), p=p, n=rng.randint(p, 2 * p),
                    s=rng.randint(2, 8))
    if kind == "learn":
        p, n, s = GROUPS[rng.choice([8, 12, 16])]
        return dict(kind="learn", N=_log(rng, 1500, 200000 if p < 16 else 100000), p=p, n=n, s=s)
    if kind == "update":
        p1, p2 = rng.randint(6, 16), rng.randint(6, 16)
        return dict(kind="update", N=_log(rng, 4000, 150000), p1=p1, p2=p2, n1=rng.randint(p1, 2 * p1),
                    n2=rng.randint(p2, 2 * p2), s=rng.randint(3, 8))
    if kind == "ortho":
        if rng.random() < 0.5:
            p1 = p2 = rng.choice([8, 12, 16])
        else:
            p1, p2 = rng.randint(6, 16), rng.randint(6, 16)
        return dict(kind="ortho", N=_log(rng, 2000, 200000), p1=p1, p2=p2, s=rng.randint(2, 8))
    if kind == "code3":
        if rng.random() < 0.5:
            return dict(kind="code3", N=_log(rng, 2000, 50000), p1=4, p2=4, p3=16, n1=8, n2=8, n3=16, s=8)
        p1, p2, p3 = rng.randint(2, 5), rng.randint(2, 5), rng.randint(4, 12)
        return dict(kind="code3", N=_log(rng, 1000, 10000), p1=p1, p2=p2, p3=p3, n1=p1 + rng.randint(0, p1),
                    n2=p2 + rng.randint(0, p2), n3=min(p3 + 2, 12), s=rng.randint(2, 6))
    if kind == "train":
        p, n, s = GROUPS[rng.choice([8, 12])]
        b = 8 * _log(rng, 64, 512)
        return dict(kind="train", N=b * rng.randint(2, 8), batch=b, p=p, n=n, s=s, hidden=8 * rng.randint(16, 64))
    p, n, s = GROUPS[rng.choice([8, 12])]
    return dict(kind="learned", N=_log(rng, 5000, 200000 if p == 8 else 60000), p=p, n=n, s=s,
                k=rng.choice([16, 24, 32]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _unit(D):
    return D / D.norm(dim=0, keepdim=True)


def _dct(p, n):
    """Overcomplete cosine dictionary, columns of unit norm (the usual start in patch denoising)."""
    a = torch.arange(p, device=DEV, dtype=torch.float64)[:, None]
    k = torch.arange(n, device=DEV, dtype=torch.float64)[None, :]
    return _unit(torch.cos(math.pi * (a + 0.5) * k / n)).float()


def _image(g, H, W):
    """Regions with intensity ramps, and texture, range 0..255."""
    yy = torch.arange(H, device=DEV).float()[:, None]
    xx = torch.arange(W, device=DEV).float()[None, :]
    c = _rand(g, 24, 5)
    d = (yy - c[:, 0, None, None] * H) ** 2 + (xx - c[:, 1, None, None] * W) ** 2
    lab = d.argmin(dim=0)
    img = 40 + 175 * c[lab, 2] + 0.3 * (c[lab, 3] - 0.5) * (yy - H / 2) + 0.3 * (c[lab, 4] - 0.5) * (xx - W / 2)
    f = torch.sqrt(torch.fft.fftfreq(H, device=DEV)[:, None] ** 2 + torch.fft.fftfreq(W, device=DEV)[None, :] ** 2)
    f[0, 0] = 1.0
    spec = torch.fft.fft2(_randn(g, H, W)) / f
    spec[0, 0] = 0
    tex = torch.fft.ifft2(spec).real
    return (img + tex * (6.0 / tex.std())).clamp(0.0, 255.0)


def _patches(g, N, p1, p2):
    """N mean-removed patches at random places of four 512 x 512 images."""
    imgs = torch.stack([_image(g, 512, 512) for _ in range(4)])
    win = imgs.unfold(1, p1, 1).unfold(2, p2, 1)
    pick = [torch.randint(0, win.shape[d], (N,), generator=g, device=DEV) for d in range(3)]
    Y = win[pick[0], pick[1], pick[2]]
    return Y - Y.mean(dim=(1, 2), keepdim=True)


def _planted(g, N, D, s, snr_db=20.0):
    """Signals sum_l x_l d1 o d2 (o d3) + noise; returns (Y, supports, coefficients)."""
    n = [d.shape[1] for d in D]
    q = torch.randint(0, math.prod(n), (N, s), generator=g, device=DEV)
    x = _randn(g, N, s)
    i = [q % n[0], (q // n[0]) % n[1]] + ([q // (n[0] * n[1])] if len(D) == 3 else [])
    F = [d.t()[k] for d, k in zip(D, i)]                       # (N, s, p_m)
    if len(D) == 2:
        Y = torch.bmm((F[0] * x[..., None]).transpose(1, 2), F[1])
    else:
        ab = (F[0][..., :, None] * F[1][..., None, :] * x[..., None, None]).flatten(2)
        Y = torch.bmm(ab.transpose(1, 2), F[2]).view(N, F[0].shape[2], F[1].shape[2], F[2].shape[2])
    e = Y.flatten(1).pow(2).mean(dim=1).sqrt() * 10.0 ** (-snr_db / 20.0)
    return Y + _randn(g, *Y.shape) * e.view(-1, *([1] * (Y.dim() - 1))), q, x


def _hyper(g, N, p1, p2):
    """Mixtures of 8 smooth spectra at 30 dB (pixels x bands)."""
    b = torch.arange(p2, device=DEV).float()
    c = _rand(g, 8, 3, 3)
    S = ((0.2 + 0.8 * c[..., 2, None]) * torch.exp(-0.5 * ((b - c[..., 0, None] * p2) /
                                                           (p2 / 16 + c[..., 1, None] * p2 * 3 / 16)) ** 2)).sum(1)
    A = -torch.log(_rand(g, N, p1, 8).clamp_min(1e-12))
    Y = (A / A.sum(2, keepdim=True)) @ S
    e = Y.flatten(1).pow(2).mean(dim=1).sqrt() * 10.0 ** (-30.0 / 20.0)
    return Y + _randn(g, N, p1, p2) * e[:, None, None]


def _inputs(case, seed):
    """The tensors of a case (mathematical layout), from the seed alone."""
    g = _gen(seed)
    k = case["kind"]
    if k == "code":
        p1, p2, n1, n2, N = case["p1"], case["p2"], case["n1"], case["n2"], case["N"]
        D1, D2 = _unit(_randn(g, p1, n1)), _unit(_randn(g, p2, n2))
        if case["data"] == "patches":
            return dict(Y=_patches(g, N, p1, p2), D1=D1, D2=D2)
        if case["data"] == "hyper":
            return dict(Y=_hyper(g, N, p1, p2), D1=D1, D2=D2)
        Y, _, _ = _planted(g, N, (D1, D2), case["s"])
        # the dictionaries in hand are near those that made the signals, as learned ones are
        return dict(Y=Y, D1=_unit(D1 + 0.1 * _unit(_randn(g, p1, n1))), D2=_unit(D2 + 0.1 * _unit(_randn(g, p2, n2))))
    if k == "learn":
        p, n, N = case["p"], case["n"], case["N"]
        return dict(Y=_patches(g, N, p, p), D1=_unit(_randn(g, p, n)), D2=_unit(_randn(g, p, n)))
    if k == "batch":
        img = _image(g, case["H"], case["W"])
        return dict(image=img + case["sigma"] * _randn(g, case["H"], case["W"]))
    if k == "io":
        H, W, p, n, s = (case[v] for v in ("H", "W", "p", "n", "s"))
        N = (H - p + 1) * (W - p + 1)
        nnz = (torch.log(_rand(g, N).clamp_min(1e-9)) / math.log(0.45)).long().clamp_max(s)
        q = torch.randint(0, n * n, (N, s), generator=g, device=DEV)
        on = torch.arange(s, device=DEV)[None, :] < nnz[:, None]
        return dict(image=_image(g, H, W), means=255.0 * _rand(g, N), nnz=nnz.int(),
                    support=torch.where(on, q, -1).int(), coef=torch.where(on, 30.0 * _randn(g, N, s), 0.0),
                    D1=_unit(_randn(g, p, n)), D2=_unit(_randn(g, p, n)))
    if k == "update":
        p1, p2, n1, n2, N, s = (case[v] for v in ("p1", "p2", "n1", "n2", "N", "s"))
        D1, D2 = _unit(_randn(g, p1, n1)), _unit(_randn(g, p2, n2))
        Y, q, x = _planted(g, N, (D1, D2), s)
        return dict(Y=Y, support=q.int(), coef=x * (1.0 + 0.05 * _randn(g, N, s)), nnz=torch.full((N,), s, device=DEV).int(),
                    D1=_unit(D1 + 0.1 * _unit(_randn(g, p1, n1))), D2=_unit(D2 + 0.1 * _unit(_randn(g, p2, n2))))
    if k == "ortho":
        p1, p2 = case["p1"], case["p2"]
        Q = [torch.linalg.qr(_randn(g, p, p).double().cpu())[0].float().to(DEV) for p in (p1, p2)]
        return dict(Y=_patches(g, case["N"], p1, p2), D1=Q[0], D2=Q[1])
    if k == "code3":
        D = [_unit(_randn(g, case["p%d" % m], case["n%d" % m])) for m in (1, 2, 3)]
        Y, _, _ = _planted(g, case["N"], D, case["s"])
        return dict(Y=Y, D1=D[0], D2=D[1], D3=D[2])
    # train, learned: signals of the planted model with its supports as labels
    p, n, N = case["p"], case["n"], case["N"]
    D1, D2 = _unit(_randn(g, p, n)), _unit(_randn(g, p, n))
    Y, q, _ = _planted(g, N, (D1, D2), case["s"])
    d = dict(Y=Y, D1=D1, D2=D2, support=q.int())
    if k == "train":
        h, P, Q = case["hidden"], p * p, n * n
        d.update(W1=_randn(g, h, P) * math.sqrt(2.0 / P), b1=torch.zeros(h, device=DEV),
                 W2=_randn(g, Q, h) * math.sqrt(1.0 / h), b2=torch.full((Q,), -3.0, device=DEV))
    else:
        # a network that scores a pair by how strongly the signal correlates with it:
        # two hidden units per pair (its atom and the negative), as a trained one tends to
        K = torch.einsum("ai,bj->jiba", D1, D2).reshape(n * n, p * p)
        K = K + 0.02 * _randn(g, *K.shape)
        eye = torch.eye(n * n, device=DEV)
        d.update(W1=3.0 * torch.cat([K, -K]), b1=torch.zeros(2 * n * n, device=DEV), W2=torch.cat([eye, eye], dim=1),
                 b2=torch.zeros(n * n, device=DEV))
    return d


_ctx = None


def _context():
    """One library context for the program, as the framework's own drivers hold it."""
    global _ctx
    if _ctx is None:
        _ctx = sdl.Context(0)
    return _ctx


def prepare(case, seed):
    d = _inputs(case, seed)
    k = case["kind"]
    st = dict(case=case, ctx=_context())
    for m in ("D1", "D2", "D3"):
        if m in d:
            st[m] = sdl.dictionary(d[m])
    if k == "batch":
        specs = []
        for p in (int(v) for v in case["groups"].split(",")):
            p, n, s = GROUPS[p]
            w = d["image"].unfold(0, p, 1).unfold(1, p, 1).reshape(-1, p, p)
            Y = sdl.signals(w - w.mean(dim=(1, 2), keepdim=True))
            D = sdl.dictionary(_dct(p, n))
            specs.append(dict(Y=Y, D1=D, D2=D.t().contiguous().t(), s=s, eps=1.15 * case["sigma"] * p))
        st["batch"] = sdl.Batch(st["ctx"], specs)
        return st
    if k == "io":
        st.update(image=d["image"], means=d["means"], codes=sdl.Codes(d["support"], d["coef"], d["nnz"]))
        return st
    st["Y"] = sdl.signals3(d["Y"]) if k == "code3" else sdl.signals(d["Y"])
    if k == "update":
        st["codes"] = sdl.Codes(d["support"], d["coef"], d["nnz"])
    elif k in ("learn", "ortho"):
        st["codes"] = sdl.Codes.empty(case["N"], case["s"], DEV)
    elif k in ("train", "learned"):
        p, n = case["p"], case["n"]
        st["mlp"] = sdl.MLP(st["ctx"], p, p, n, n, hidden=d["W1"].shape[0], max_batch=case.get("batch", 4096))
        st["mlp"].set_weights(*(d[w].cpu().numpy() for w in ("W1", "b1", "W2", "b2")))
        st["labels"] = sdl.Codes(d["support"], None, None)
    return st


def _codes(c):
    return dict(support=c.support, coef=c.coef, nnz=c.nnz, res_energy=c.res_energy)


def run(st):
    case, ctx = st["case"], st["ctx"]
    k = case["kind"]
    if k == "code":
        return _codes(ctx.sparse_code(st["Y"], st["D1"], st["D2"], case["s"]))
    if k == "batch":
        st["batch"].sparse_code()
        return [_codes(g["codes"]) for g in st["batch"].groups]
    if k == "io":
        patches, means = sdl.extract_patches(st["image"], case["p"])
        image = sdl.patch_average(ctx, st["codes"], st["means"], st["D1"], st["D2"], case["p"], case["H"], case["W"])
        return dict(patches=patches, means=means, image=image)
    if k == "learn":
        c = ctx.iterate(st["Y"], st["D1"], st["D2"], case["s"], out=st["codes"])
        return dict(D1=st["D1"], D2=st["D2"], support=c.support, coef=c.coef, nnz=c.nnz)
    if k == "update":
        ctx.update_D1(st["Y"], st["D1"], st["D2"], st["codes"])
        ctx.update_D2(st["Y"], st["D1"], st["D2"], st["codes"])
        return dict(D1=st["D1"], D2=st["D2"], coef=st["codes"].coef)
    if k == "ortho":
        c = ctx.ortho_iterate(st["Y"], st["D1"], st["D2"], case["s"], out=st["codes"])
        return dict(D1=st["D1"], D2=st["D2"], support=c.support, coef=c.coef, nnz=c.nnz)
    if k == "code3":
        return _codes(ctx.sparse_code3(st["Y"], st["D1"], st["D2"], st["D3"], case["s"]))
    if k == "train":
        loss = learned.train(st["mlp"], st["Y"], st["labels"], epochs=1, batch=case["batch"])
        W1, b1, W2, b2 = st["mlp"].get_weights()
        return dict(loss=np.array(loss, dtype=np.float32), W1=W1, b1=b1, W2=W2, b2=b2)
    c, flags, nfb, guard = st["mlp"].sparse_code(st["Y"], st["D1"], st["D2"], case["s"], k=case["k"])
    return dict(_codes(c), flags=flags, n_fallback=nfb, guard=guard)


# ------------------------------------------------------------------ work
def _code_flops(p1, p2, n1, n2, s):
    """Correlations in the cheaper order, one rank-one update per earlier pick and step, the scan."""
    c0 = 2 * min(p1 * p2 * n2 + n1 * p1 * n2, n1 * p1 * p2 + n1 * p2 * n2)
    return c0 + n1 * n2 * s * (s - 1) + n1 * n2 * s


def _sum_flops(p1, p2, s):
    """Both sides' sums of one signal: every pick's projection, every pair of picks."""
    return 2 * s * (2 * p1 * p2 + p1 + p2) + 2 * 3 * s * s


def work(case):
    k = case["kind"]
    if k == "batch":
        b = f = 0
        for p in (int(v) for v in case["groups"].split(",")):
            p, n, s = GROUPS[p]
            N = (case["H"] - p + 1) * (case["W"] - p + 1)
            b += N * (4 * p * p + 8 * s + 8)
            # most patches are within the error target after no or one pick
            f += N * (2 * p * p + 0.3 * _code_flops(p, p, n, n, 1))
        return dict(bytes=b, flops=f)
    if k == "io":
        p, s = case["p"], case["s"]
        N = (case["H"] - p + 1) * (case["W"] - p + 1)
        return dict(bytes=4 * N * p * p + N * (8 * s + 8) + 8 * case["H"] * case["W"], flops=N * p * p * 5)
    N, s = case["N"], case["s"]
    if k in ("learn", "learned", "train"):
        p1 = p2 = case["p"]
        n1 = n2 = case["n"]
    elif k == "ortho":
        p1, p2 = n1, n2 = case["p1"], case["p2"]
    else:
        p1, p2, n1, n2 = case["p1"], case["p2"], case["n1"], case["n2"]
    if k == "code":
        return dict(bytes=N * (4 * p1 * p2 + 8 * s + 8), flops=N * _code_flops(p1, p2, n1, n2, s))
    if k == "learn":
        return dict(bytes=N * (2 * 4 * p1 * p2 + 8 * s + 4),
                    flops=N * (2 * _code_flops(p1, p2, n1, n2, s) + _sum_flops(p1, p2, s)))
    if k == "update":
        return dict(bytes=N * (2 * 4 * p1 * p2 + 2 * 12 * s), flops=N * _sum_flops(p1, p2, s))
    if k == "ortho":
        c0 = 2 * (p1 * p2 * p2 + p1 * p1 * p2)
        return dict(bytes=N * (2 * 4 * p1 * p2 + 8 * s + 4), flops=N * 2 * (c0 + p1 * p2 * s + 4 * s * (p1 + p2)))
    if k == "code3":
        p3, n3 = case["p3"], case["n3"]
        c0 = 2 * (n1 * p1 * p2 * p3 + n1 * n2 * p2 * p3 + n1 * n2 * n3 * p3)
        return dict(bytes=N * (4 * p1 * p2 * p3 + 8 * s + 8), flops=N * (c0 + n1 * n2 * n3 * s * s))
    P, Q = p1 * p2, n1 * n2
    if k == "train":
        h = case["hidden"]
        steps = N // case["batch"]
        w = h * P + Q * h + h + Q
        return dict(bytes=N * (4 * P + 4 * s) + steps * 24 * w + 4 * w, flops=N * (2 * (h * P + Q * h) * 2 + 2 * Q * h))
    return dict(bytes=N * (4 * P + 8 * s + 12), flops=N * (2 * 2 * Q * (P + Q) + _code_flops(p1, p2, n1, n2, s)))


# ------------------------------------------------------------------ 64 bits
def _chunks(N, width):
    step = max(1, min(N, (1 << 27) // max(1, width)))
    return [slice(a, min(N, a + step)) for a in range(0, N, step)]


def _omp64(Y, D, s, eps2=0.0):
    """Greedy pursuit over the tuples of atoms of two or three dictionaries: (q (N, s), x (N, s), energy (N,))."""
    G = [d.t() @ d for d in D]
    n = [d.shape[1] for d in D]
    Q, N = math.prod(n), Y.shape[0]
    q_all = torch.full((N, s), -1, dtype=torch.int64, device=DEV)
    x_all = torch.zeros(N, s, dtype=torch.float64, device=DEV)
    e_all = torch.zeros(N, dtype=torch.float64, device=DEV)

    def parts(q):
        return [q % n[0], (q // n[0]) % n[1]] + ([q // (n[0] * n[1])] if len(D) == 3 else [])

    for sl in _chunks(N, 3 * Q):
        y = Y[sl]
        m = y.shape[0]
        if len(D) == 2:
            C0 = (D[0].t() @ y @ D[1]).transpose(1, 2).reshape(m, Q)
        else:
            C0 = torch.einsum("klba,ai->klbi", torch.einsum("kabc,cl->klba", y, D[2]), D[0])
            C0 = torch.einsum("klbi,bj->klji", C0, D[1]).reshape(m, Q)
        E = y.flatten(1).pow(2).sum(1)
        q = torch.full((m, s), -1, dtype=torch.int64, device=DEV)
        L = torch.zeros(m, s, s, dtype=torch.float64, device=DEV)
        yv = torch.zeros(m, s, dtype=torch.float64, device=DEV)
        x = torch.zeros(m, s, dtype=torch.float64, device=DEV)
        picked = torch.zeros(m, Q, dtype=torch.bool, device=DEV)
        live = torch.ones(m, dtype=torch.bool, device=DEV)
        for t in range(s):
            if eps2 > 0:
                live = live & (E > eps2)
            sc = C0
            if t:
                R = [g[i] for g, i in zip(G, parts(q[:, :t].clamp_min(0)))]      # (m, t, n_k)
                R[0] = R[0] * x[:, :t, None]
                U = R[1] if len(D) == 2 else (R[2][..., :, None] * R[1][..., None, :]).flatten(2)
                sc = C0 - torch.bmm(U.transpose(1, 2), R[0]).reshape(m, Q)
            sc = sc.abs().masked_fill(picked, -1.0)
            best, qt = sc.max(dim=1)
            live = live & (best > 0)
            it = parts(qt)
            A = torch.ones(m, t + 1, dtype=torch.float64, device=DEV)
            for g, i, j in zip(G, it, parts(torch.cat([q[:, :t].clamp_min(0), qt[:, None]], 1))):
                A = A * g[i[:, None], j]
            w = torch.zeros(m, t, dtype=torch.float64, device=DEV)
            for r in range(t):
                w[:, r] = (A[:, r] - (L[:, r, :r] * w[:, :r]).sum(1)) / L[:, r, r]
            d = A[:, t] - (w * w).sum(1)
            live = live & (d > 1e-6 * A[:, t])
            Ltt = d.clamp_min(1e-300).sqrt()
            yt = (C0.gather(1, qt[:, None])[:, 0] - (w * yv[:, :t]).sum(1)) / Ltt
            L[:, t, :t] = w
            L[:, t, t] = torch.where(live, Ltt, torch.ones_like(Ltt))
            yv[:, t] = yt
            xn = torch.zeros(m, s, dtype=torch.float64, device=DEV)
            for r in range(t, -1, -1):
                xn[:, r] = (yv[:, r] - (L[:, r + 1:t + 1, r] * xn[:, r + 1:t + 1]).sum(1)) / L[:, r, r]
            x = torch.where(live[:, None], xn, x)
            q[:, t] = torch.where(live, qt, q[:, t])
            picked.scatter_(1, qt[:, None], True)
            E = torch.where(live, E - yt * yt, E)
        q_all[sl], x_all[sl], e_all[sl] = q, x, E.clamp_min(0.0)
    return q_all, x_all, e_all


def _update64(Y, D1, D2, q, x, side):
    """Least-squares update of one dictionary with the codes fixed: (D with unit columns, norms)."""
    n1, n2 = D1.shape[1], D2.shape[1]
    D = D1 if side == 1 else D2
    P = torch.zeros(D.shape[1], D.shape[1], dtype=torch.float64, device=DEV)
    B = torch.zeros(D.shape[0], D.shape[1], dtype=torch.float64, device=DEV)
    for sl in _chunks(Y.shape[0], 4 * n1 * n2):
        m = q[sl].shape[0]
        X = torch.zeros(m, n1 * n2, dtype=torch.float64, device=DEV)
        X.scatter_add_(1, q[sl].clamp_min(0), torch.where(q[sl] >= 0, x[sl], 0.0))
        X = X.view(m, n2, n1)                                            # X[k, j, i]
        if side == 1:
            T = (X.transpose(1, 2) @ D2.t()).transpose(1, 2)             # (m, p2, n1)
            Z = Y[sl].transpose(1, 2)                                    # (m, p2, p1)
        else:
            T = (X @ D1.t()).transpose(1, 2)                             # (m, p1, n2)
            Z = Y[sl]                                                    # (m, p1, p2)
        T = T.reshape(-1, T.shape[2])
        P += T.t() @ T
        B += Z.reshape(-1, Z.shape[2]).t() @ T
    on = P.diagonal() > 0
    Dn = D.clone()
    Dn[:, on] = torch.linalg.solve(P[on][:, on], B[:, on].t()).t()
    norm = torch.where(on, Dn.norm(dim=0), 1.0)
    return Dn / norm, norm


def exact(case, seed):
    k = case["kind"]
    d = {v: t.double() if t.is_floating_point() else t.long() for v, t in _inputs(case, seed).items()}
    if k == "code":
        q, x, e = _omp64(d["Y"], (d["D1"], d["D2"]), case["s"])
        return dict(support=None, coef=x, nnz=None, res_energy=e)
    if k == "code3":
        q, x, e = _omp64(d["Y"], (d["D1"], d["D2"], d["D3"]), case["s"])
        return dict(support=None, coef=x, nnz=None, res_energy=e)
    if k == "batch":
        out = []
        for p in (int(v) for v in case["groups"].split(",")):
            p, n, s = GROUPS[p]
            w = d["image"].float().unfold(0, p, 1).unfold(1, p, 1).reshape(-1, p, p)
            Y = (w - w.mean(dim=(1, 2), keepdim=True)).double()
            D = _dct(p, n).double()
            q, x, e = _omp64(Y, (D, D), s, eps2=(1.15 * case["sigma"] * p) ** 2)
            out.append(dict(support=None, coef=x, nnz=None, res_energy=e))
        return out
    if k == "io":
        p, n, s, H, W = (case[v] for v in ("p", "n", "s", "H", "W"))
        w = d["image"].unfold(0, p, 1).unfold(1, p, 1).reshape(-1, p, p)
        means = w.mean(dim=(1, 2))
        q, x = d["support"].clamp_min(0), d["coef"]
        rec = torch.bmm((d["D1"].t()[q % n] * x[..., None]).transpose(1, 2), d["D2"].t()[q // n]) + d["means"][:, None, None]
        acc = torch.zeros(H, W, dtype=torch.float64, device=DEV)
        cnt = torch.zeros_like(acc)
        rec = rec.view(H - p + 1, W - p + 1, p, p)
        for a in range(p):
            for b in range(p):
                acc[a:a + H - p + 1, b:b + W - p + 1] += rec[:, :, a, b]
                cnt[a:a + H - p + 1, b:b + W - p + 1] += 1
        return dict(patches=w - means[:, None, None], means=means, image=acc / cnt)
    if k == "learn":
        Y, D1, D2, s = d["Y"], d["D1"], d["D2"], case["s"]
        q, x, _ = _omp64(Y, (D1, D2), s)
        D1, _ = _update64(Y, D1, D2, q, x, 1)
        q, x, _ = _omp64(Y, (D1, D2), s)
        D2, norm = _update64(Y, D1, D2, q, x, 2)
        return dict(D1=D1, D2=D2, support=None, coef=x * norm[q.clamp_min(0) // case["n"]], nnz=None)
    if k == "update":
        n1 = case["n1"]
        D1, D2, q, x = d["D1"], d["D2"], d["support"], d["coef"]
        D1, norm = _update64(d["Y"], D1, D2, q, x, 1)
        x = x * norm[q % n1]
        D2, norm = _update64(d["Y"], D1, D2, q, x, 2)
        return dict(D1=D1, D2=D2, coef=x * norm[q // n1])
    if k == "ortho":
        D = [d["D1"], d["D2"]]
        x = None
        for side in (0, 1):
            B = torch.zeros_like(D[side])
            xs = []
            for sl in _chunks(case["N"], 4 * case["p1"] * case["p2"]):
                y = d["Y"][sl]
                C = (D[0].t() @ y @ D[1]).transpose(1, 2).flatten(1)
                q = C.abs().topk(case["s"], dim=1).indices
                xs.append(C.gather(1, q))
                X = torch.zeros_like(C).scatter_(1, q, xs[-1]).view(-1, case["p2"], case["p1"]).transpose(1, 2)
                if side == 0:
                    B += torch.einsum("kab,kib->ai", y @ D[1], X)
                else:
                    B += torch.einsum("kab,kaj->bj", y, D[0] @ X)
            U, _, Vh = torch.linalg.svd(B)
            D[side] = U @ Vh
            x = torch.cat(xs)
        return dict(D1=D[0], D2=D[1], support=None, coef=x, nnz=None)
    if k == "train":
        P = [d[w].clone() for w in ("W1", "b1", "W2", "b2")]
        M = [torch.zeros_like(w) for w in P]
        V = [torch.zeros_like(w) for w in P]
        N, B, Q = case["N"], case["batch"], case["n"] ** 2
        X = d["Y"].transpose(1, 2).flatten(1)
        X = X / X.norm(dim=1, keepdim=True)
        losses = []
        for step, a in enumerate(range(0, N - B + 1, B), 1):
            ps = [w.detach().requires_grad_() for w in P]
            t = torch.zeros(B, Q, dtype=torch.float64, device=DEV).scatter_(1, d["support"][a:a + B], 1.0)
            z = torch.nn.functional.gelu(X[a:a + B] @ ps[0].t() + ps[1]) @ ps[2].t() + ps[3]
            loss = (torch.nn.functional.softplus(z) - t * z).sum(1).mean()
            grads = torch.autograd.grad(loss, ps)
            losses.append(loss.item())
            for i, g in enumerate(grads):
                M[i] = 0.9 * M[i] + 0.1 * g
                V[i] = 0.999 * V[i] + 0.001 * g * g
                P[i] = P[i] - 2e-3 * (M[i] / (1 - 0.9 ** step)) / ((V[i] / (1 - 0.999 ** step)).sqrt() + 1e-8)
        P = [w.cpu().numpy() for w in P]
        return dict(loss=np.array([np.mean(losses)]), W1=P[0], b1=P[1], W2=P[2], b2=P[3])
    return None   # learned: what is coded again depends on 16-bit scores
