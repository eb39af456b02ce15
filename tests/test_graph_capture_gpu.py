"""The entry points whose kernels are dependent launches, captured in a CUDA
graph and replayed with new inputs in the same buffers: the bits of the eager
call.  Two calls per capture, so that a call's first kernel also follows the
last one of another."""
import numpy as np
import pytest

import svdlut_inputs as si

pytestmark = pytest.mark.gpu


def _captured(fn, fill, n_inputs=3):
    """fn() -> list of tensors (fresh or the same buffers); fill(k) writes input
    set k into the inputs.  Compares a replayed graph of two calls with eager calls."""
    import torch
    eager = []
    for k in range(n_inputs):
        fill(k)
        eager.append([t.clone() for t in fn()])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        fn()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        first, second = fn(), fn()
    for k in range(n_inputs):
        fill(k)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        for got in (first, second):
            for a, r in zip(got, eager[k]):
                assert torch.equal(a, r), k


def _sv():
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    return torch, sv


@pytest.mark.parametrize("B,H,W", [(2, 70, 130), (20, 64, 60), (1, 600, 900)])
def test_backward(B, H, W):
    torch, sv = _sv()
    d = si.spatial_dims(H, W)
    sets = []
    for k in range(3):
        x, p = si.make_batch(1600 + k, B, H, W, d)
        sets.append((torch.from_numpy(x).cuda(), sv.to_device(p), torch.from_numpy(si.make_upstream(1610 + k, x.shape)).cuda()))
    x, p, dy = sets[0][0].clone(), {n: t.clone() for n, t in sets[0][1].items()}, sets[0][2].clone()

    def fill(k):
        x.copy_(sets[k][0])
        dy.copy_(sets[k][2])
        for n in p:
            p[n].copy_(sets[k][1][n])

    def fn():
        y = sv.apply(x, p)
        return [y] + list(sv.backward(x, p, dy).values())

    _captured(fn, fill)


def test_losses():
    torch, sv = _sv()
    g = torch.Generator(device="cuda").manual_seed(3)
    sets = [torch.rand(2, 3, 3, 90, 84, device="cuda", generator=g) for _ in range(3)]
    y, t = torch.empty(3, 3, 90, 84, device="cuda"), torch.empty(3, 3, 90, 84, device="cuda")

    def fill(k):
        y.copy_(sets[k][0])
        t.copy_(sets[k][1])

    def fn():
        dy = torch.empty_like(y)
        a = sv.mse(y, t, dy=dy)
        b = sv.cie94(y, t, weight=0.01, dy=dy, accumulate=True)
        return [a, b, dy]

    _captured(fn, fill)


@pytest.mark.parametrize("B", [1, 5])
def test_generator(B):
    torch, sv = _sv()
    K, H, W = 6, 300, 280
    gen = torch.Generator(device="cuda").manual_seed(4)
    n = int(sv._lib.load().svdlut_generator_param_count(K))
    weights = [0.1 * torch.randn(n, device="cuda", generator=gen) for _ in range(3)]
    images = [torch.rand(B, 3, H, W, device="cuda", generator=gen) for _ in range(3)]
    G = sv.Generator(K, weights[0].clone(), max_batch=B)
    x = images[0].clone()
    up = {k: torch.randn(v.shape, device="cuda", generator=gen) for k, v in G.empty_params(B).items()}

    def fill(k):
        x.copy_(images[k])
        G.weights.copy_(weights[k])

    def fn():
        out = G.forward(x, training=True, seed=7)
        return list(out.values()) + [G.backward(up)]

    _captured(fn, fill)


def test_photos_and_3d_lut():
    torch, sv = _sv()
    H, W = 520, 514
    d = si.paper_dims()
    codes = [si.make_image_u16(np.random.default_rng(1700 + k), H, W) for k in range(3)]
    photos = [torch.from_numpy(c[None]).cuda() for c in codes]
    images = [torch.from_numpy((c / 65535.0).astype(np.float32)).cuda() for c in codes]
    _, p = si.make_batch(1701, 1, H, W, d)
    pd = sv.to_device(p)
    lut = torch.from_numpy(si.make_lut3d(np.random.default_rng(1702), 17, "photo").astype(np.float32)).cuda()
    x16, xf = photos[0].clone(), images[0].clone()

    def fill(k):
        x16.copy_(photos[k])
        xf.copy_(images[k])

    def fn():
        return [sv.apply_io(x16, pd, "u16", "f32"), sv.lut3d_apply(xf, lut)]

    _captured(fn, fill)
