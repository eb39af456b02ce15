"""Performance cases of the SVDLUT framework: what its users have it do, timed
through the public calls of paper_2508_16121_gb300.

A photo or video pipeline calls the fused transform on frames of every size,
from thumbnails to 4K, in float, 8-bit and 16-bit formats, one by one or as a
ragged batch; a trainer calls the adjoint, the loss and the factor generator on
batches of 256 x 256 crops; a server calls the generator on full frames.

Inputs are drawn on the GPU from a seed: `mix` images are 64 x 64 tiles of
noise and of smooth gradients in turn, `photo` images are smooth gradients
under a random exposure, colour cast and gamma with mild noise.  Factors are
the identity transform plus noise.
"""
import math

import numpy as np
import torch

import paper_2508_16121_gb300 as svdlut

DT, RANK, DSC = 33, 8, 17  # LUT vertices per axis, SVD rank, intensity vertices of the grids
VIDEO_SIZES = ((640, 480), (1280, 720), (1920, 1080), (2560, 1440), (3840, 2160))
GEN_CHANNELS, GEN_HIDDEN, GEN_THUMB = (3, 8, 16, 32, 64, 64), 8, 256
CIE94_WEIGHT = 0.005


def listed():
    return [
        # a preview thumbnail with the paper's own grids (6 grids of 17^3): the smallest call,
        # where launches, host work and the tables' setup count
        {"name": "apply_f32_256", "kind": "apply", "fmt": "f32", "B": 1, "H": 256, "W": 256, "grids": "paper",
         "mode": "photo"},
        # a cropped photo of odd size (no vector accesses), grids at 1/8 resolution
        {"name": "apply_f32_odd", "kind": "apply", "fmt": "f32", "B": 1, "H": 853, "W": 1279, "grids": "eighth",
         "mode": "mix"},
        # one 4K frame, grids at 1/8 resolution: the headline workload
        {"name": "apply_f32_4k", "kind": "apply", "fmt": "f32", "B": 1, "H": 2160, "W": 3840, "grids": "eighth",
         "mode": "mix"},
        # a short burst of 8-bit 1080p video frames
        {"name": "apply_u8_4x1080p", "kind": "apply", "fmt": "u8", "B": 4, "H": 1080, "W": 1920, "grids": "eighth",
         "mode": "mix"},
        # tone mapping of a 16-bit interleaved 4K photo to 8 bits
        {"name": "apply_u16hwc_4k", "kind": "apply", "fmt": "u16_hwc", "B": 1, "H": 2160, "W": 3840, "grids": "paper",
         "mode": "mix"},
        # a queue of frames of 480p to 4K in one launch (46 Mpx)
        {"name": "ragged_16", "kind": "ragged", "fmt": "f32", "n": 16, "sizes": "video", "sizes_seed": 16123,
         "mode": "mix"},
        # every gradient of a batch of 1080p frames (fine-tuning factors on full frames)
        {"name": "backward_8x1080p", "kind": "backward", "B": 8, "H": 1080, "W": 1920, "grids": "eighth",
         "mode": "mix"},
        # the parameter gradients of a training batch of crops
        {"name": "backward_64x256", "kind": "backward", "B": 64, "H": 256, "W": 256, "grids": "generated",
         "mode": "photo"},
        # the learned factors of four 4K frames (serving)
        {"name": "generate_4x4k", "kind": "generate", "B": 4, "H": 2160, "W": 3840, "K": 8},
        # the loss of a training batch and its gradient (MSE + 0.005 CIE94)
        {"name": "loss_64x256", "kind": "loss", "B": 64, "H": 256, "W": 256},
        # a training step up to the weight gradients: generator, transform, loss and their gradients
        {"name": "train_64x256", "kind": "train", "B": 64, "H": 256, "W": 256, "K": 8},
        # a 3D LUT applied to a 4K frame
        {"name": "lut3d_4k", "kind": "lut3d", "B": 1, "H": 2160, "W": 3840, "D": 33, "mode": "mix"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _frame(rng, most):
    """H, W of a frame of at most `most` pixels, odd ones among them."""
    while True:
        H, W = _log(rng, 64, 2160), _log(rng, 64, 3840)
        if rng.random() < 0.5:
            W = max(64, W // 8 * 8)
        if H * W <= most and 1 / 4 <= W / H <= 4:
            return H, W


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "ragged", "backward", "backward", "generate", "loss", "train", "lut3d"))
    mode = rng.choice(("mix", "photo"))
    grids = rng.choice(("eighth", "paper", "generated"))
    if kind == "apply":
        H, W = _frame(rng, 3840 * 2160)
        B = max(1, min(_log(rng, 1, 80), 16_000_000 // (H * W)))
        return {"kind": kind, "fmt": rng.choice(("f32", "f32", "u8", "u8_hwc", "u16", "u16_hwc")), "B": B, "H": H,
                "W": W, "grids": grids, "mode": mode}
    if kind == "ragged":
        return {"kind": kind, "fmt": rng.choice(("f32", "u8")), "n": _log(rng, 2, 16), "sizes": "any",
                "sizes_seed": rng.randrange(1 << 20), "mode": mode}
    if kind == "backward":
        H, W = _frame(rng, 1920 * 1080)
        B = max(1, min(_log(rng, 1, 64), 8_000_000 // (H * W)))
        return {"kind": kind, "B": B, "H": H, "W": W, "grids": grids, "mode": mode}
    if kind == "generate":
        H, W = _frame(rng, 3840 * 2160)
        B = max(1, min(_log(rng, 1, 64), 32_000_000 // (H * W)))
        return {"kind": kind, "B": B, "H": H, "W": W, "K": rng.choice((6, 8))}
    if kind == "loss":
        H, W = _frame(rng, 1920 * 1080)
        B = max(1, min(_log(rng, 1, 64), 8_000_000 // (H * W)))
        return {"kind": kind, "B": B, "H": H, "W": W}
    if kind == "train":
        size = rng.choice((128, 192, 256, 320))
        return {"kind": kind, "B": min(_log(rng, 2, 64), 64 * 256 * 256 // (size * size)), "H": size, "W": size,
                "K": rng.choice((6, 8))}
    H, W = _frame(rng, 3840 * 2160)
    return {"kind": kind, "B": max(1, min(_log(rng, 1, 8), 8_000_000 // (H * W))), "H": H, "W": W,
            "D": rng.choice((17, 25, 33)), "mode": mode}


# ---------------------------------------------------------------- inputs

def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 16121)
    return g, np.random.default_rng([16121, int(seed)])


def _images(gen, B, H, W, mode):
    """[B,3,H,W] float32 in [0,1]."""
    def u(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, device="cuda", generator=gen)

    yy = torch.arange(H, device="cuda", dtype=torch.float32).view(1, 1, H, 1) / H
    xx = torch.arange(W, device="cuda", dtype=torch.float32).view(1, 1, 1, W) / W
    s = (B, 3, 1, 1)
    img = u(0.1, 0.5, *s) + u(-0.4, 0.4, *s) * xx + u(-0.4, 0.4, *s) * yy
    for _ in range(2):
        img = img + u(0.05, 0.25, *s) * torch.sin(2 * math.pi * (u(0.5, 3.0, *s) * xx + u(0.5, 3.0, *s) * yy)
                                                  + u(0.0, 2 * math.pi, *s))
    img = img.clamp(0, 1)
    if mode == "photo":
        img = img * u(0.5, 1.5, B, 1, 1, 1) * u(0.75, 1.25, *s)
        img = img.clamp(1e-6, 1) ** u(0.7, 1.4, B, 1, 1, 1)
        img = (img + 0.01 * torch.randn(B, 3, H, W, device="cuda", generator=gen)).clamp(0, 1)
    else:
        ty = torch.arange(H, device="cuda").view(H, 1) // 64
        tx = torch.arange(W, device="cuda").view(1, W) // 64
        img = torch.where((tx + ty) % 2 == 0, torch.rand(B, 3, H, W, device="cuda", generator=gen), img)
    return img.contiguous()


def _grid_dims(grids, H, W):
    """K, Dsx, Dsy."""
    if grids == "eighth":
        return 8, max(2, -(-W // 8)), max(2, -(-H // 8))
    return (6 if grids == "paper" else 8), 17, 17


def _identity():
    """Factors of the identity transform: U, S, V, lut_w."""
    U, V = np.zeros((3, 3, DT, RANK)), np.zeros((3, 3, DT, RANK))
    S, lut_w = np.zeros((3, 3, RANK)), np.zeros((3, 4))
    ramp, one = np.linspace(0.0, 1.0, DT), np.ones(DT)
    for c, uses in {0: ((0, True), (1, True)), 1: ((0, False), (2, True)), 2: ((1, False), (2, False))}.items():
        for p, alpha in uses:  # channel c is the first or the second axis of pair p
            U[c, p, :, 0], V[c, p, :, 0] = (ramp, one) if alpha else (one, ramp)
            S[c, p, 0], lut_w[c, p] = 1.0, 0.5
    return U, S, V, lut_w


def _params(rng, B, K, Dsx, Dsy):
    """Factors of B images on the GPU: the identity plus noise, random grids."""
    U, S, V, lut_w = _identity()
    p = {"U": U + rng.normal(0.0, 0.1, (B,) + U.shape), "V": V + rng.normal(0.0, 0.1, (B,) + V.shape)}
    S = np.repeat(S[None], B, 0)
    S[..., 0], S[..., 1:] = 1.0, rng.uniform(0.0, 1.0, S[..., 1:].shape)
    p["S"] = S
    w = np.repeat(lut_w[None], B, 0)
    w[..., :3] += rng.uniform(-0.05, 0.05, w[..., :3].shape)
    w[..., 3] = rng.uniform(-0.02, 0.02, w[..., 3].shape)
    p["lut_w"] = w
    p["g_xy"] = rng.random((B, K, Dsy, Dsx), dtype=np.float32)
    p["g_xc"] = rng.random((B, K, Dsx, DSC), dtype=np.float32)
    p["g_yc"] = rng.random((B, K, Dsy, DSC), dtype=np.float32)
    p["grid_w"] = rng.uniform(-0.05, 0.05, (B, K, 4))
    return {k: torch.as_tensor(p[k], dtype=torch.float32).contiguous().cuda() for k in svdlut.PARAM_NAMES}


def _encode(x, fmt):
    """float images as the pixel format fmt holds them."""
    if fmt.startswith("u16"):
        x = (x.double() ** 2.2 * 65535).round().to(torch.int32).to(torch.uint16)
    elif fmt.startswith("u8"):
        x = (x * 255).round().to(torch.uint8)
    return x.permute(0, 2, 3, 1).contiguous() if fmt.endswith("hwc") else x


OUT_FORMAT = {"u16": "f32", "u16_hwc": "u8_hwc", "u8_hwc": "u8_hwc"}


def _ragged_sizes(case):
    """(W, H) of each frame."""
    rng = np.random.default_rng(case["sizes_seed"])
    if case["sizes"] == "video":
        return [VIDEO_SIZES[i] for i in rng.integers(0, len(VIDEO_SIZES), case["n"])]
    out, left = [], 32_000_000
    for _ in range(case["n"]):
        h = int(round(math.exp(rng.uniform(math.log(64), math.log(2160)))))
        w = min(3840, max(64, int(h * rng.uniform(0.6, 2.0))))
        h = max(64, min(h, left // (w * 2)))
        left -= w * h
        out.append((w, h))
    return out


def _generator_shapes(K):
    """(name, shape) of the generator's weights in their order."""
    out = []
    for i in range(5):
        a, b = GEN_CHANNELS[i], GEN_CHANNELS[i + 1]
        out += [(f"conv{i}.w", (b, a, 3, 3)), (f"conv{i}.b", (b,))]
        if i < 4:
            out += [(f"in{i}.g", (b,)), (f"in{i}.b", (b,))]
    for h, n in (("s", K * 3 * DSC * DSC), ("sw", K * 4), ("t", 9 * RANK * (2 * DT + 1)), ("tw", 12)):
        out += [(f"h{h}.w1", (GEN_HIDDEN, 256)), (f"h{h}.b1", (GEN_HIDDEN,)), (f"h{h}.w2", (n, GEN_HIDDEN)),
                (f"h{h}.b2", (n,))]
    return out


def _generator_weights(rng, K):
    """A partly trained generator: He-scaled convolutions, last layers N(0, 0.1) around the identity factors."""
    U, S, V, lut_w = _identity()
    parts = []
    for n, s in _generator_shapes(K):
        if n.endswith(".g"):
            v = 1.0 + rng.normal(0.0, 0.05, s)
        elif n == "ht.b2":
            v = np.concatenate([U.ravel(), S.ravel(), V.ravel()])
        elif n == "htw.b2":
            v = lut_w.ravel()
        elif n.endswith(".w"):
            v = rng.normal(0.0, math.sqrt(2.0 / (s[1] * 9)), s)
        elif n.endswith(".w1"):
            v = rng.normal(0.0, math.sqrt(1.0 / s[1]), s)
        elif n.endswith(".w2"):
            v = rng.normal(0.0, 0.1, s)
        else:
            v = rng.normal(0.0, 0.02, s)
        parts.append(np.asarray(v).ravel())
    return torch.as_tensor(np.concatenate(parts), dtype=torch.float32).cuda()


def _graded(gen, x):
    """A retouched version of photos x: the ground truth of a training pair."""
    B = x.shape[0]
    gain = 0.8 + 0.4 * torch.rand(B, 3, 1, 1, device="cuda", generator=gen)
    gamma = 0.8 + 0.4 * torch.rand(B, 1, 1, 1, device="cuda", generator=gen)
    return ((x * gain).clamp(1e-4, 1) ** gamma).contiguous()


def _lut3d(rng, B, D):
    """Smooth 3D LUTs [B,3,D,D,D]: the identity plus low-frequency cosines."""
    v = np.linspace(0.0, 1.0, D)
    r, g, b = np.meshgrid(v, v, v, indexing="ij")
    out = np.empty((B, 3, D, D, D), np.float32)
    for i in range(B):
        x = np.stack([r, g, b])
        for _ in range(4):
            f, ph, a = rng.integers(1, 3, 3), rng.uniform(0, 2 * np.pi, 3), rng.uniform(-0.05, 0.05, 3)
            x = x + a[:, None, None, None] * np.cos(np.pi * (f[0] * r + f[1] * g + f[2] * b) + ph[:, None, None, None])
        out[i] = x
    return torch.as_tensor(out).cuda()


def prepare(case, seed):
    gen, rng = _rng(seed)
    kind = case["kind"]
    s = {"case": dict(case)}
    if kind == "ragged":
        xs, ps = [], []
        for W, H in _ragged_sizes(case):
            xs.append(_encode(_images(gen, 1, H, W, case["mode"]), case["fmt"])[0])
            p = _params(rng, 1, *_grid_dims("eighth", H, W))
            ps.append({k: v[0] for k, v in p.items()})
        s.update(xs=xs, params=ps, batch=svdlut.Batch(xs, ps))
        return s
    B, H, W = case["B"], case["H"], case["W"]
    if kind == "apply":
        s["x"] = _encode(_images(gen, B, H, W, case["mode"]), case["fmt"])
        s["params"] = _params(rng, B, *_grid_dims(case["grids"], H, W))
    elif kind == "backward":
        s["x"] = _images(gen, B, H, W, case["mode"])
        s["params"] = _params(rng, B, *_grid_dims(case["grids"], H, W))
        s["dy"] = torch.randn(B, 3, H, W, device="cuda", generator=gen)
    elif kind == "generate":
        s["x"] = _images(gen, B, H, W, "photo")
        s["gen"] = svdlut.Generator(case["K"], _generator_weights(rng, case["K"]), max_batch=B)
    elif kind == "loss":
        s["target"] = _images(gen, B, H, W, "photo")
        s["y"] = s["target"] + 0.05 * torch.randn(B, 3, H, W, device="cuda", generator=gen)
        s["dy"] = torch.empty_like(s["y"])
    elif kind == "train":
        s["x"] = _images(gen, B, H, W, "photo")
        s["target"] = _graded(gen, s["x"])
        s["gen"] = svdlut.Generator(case["K"], _generator_weights(rng, case["K"]), max_batch=B)
        s["dropout_seed"] = int(seed) % (1 << 20) + 1
        s["dy"] = torch.empty_like(s["x"])
    else:
        s["x"] = _images(gen, B, H, W, case["mode"])
        s["lut"] = _lut3d(rng, B, case["D"])
    return s


# ---------------------------------------------------------------- one pass

def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "apply":
        fmt = case["fmt"]
        if fmt in OUT_FORMAT:
            return svdlut.apply_io(state["x"], state["params"], fmt, OUT_FORMAT[fmt])
        return svdlut.apply(state["x"], state["params"])
    if kind == "ragged":
        return state["batch"].run()
    if kind == "backward":
        return svdlut.backward(state["x"], state["params"], state["dy"])
    if kind == "generate":
        return state["gen"].forward(state["x"])
    if kind == "loss":
        y, t, dy = state["y"], state["target"], state["dy"]
        loss = svdlut.mse(y, t, dy)
        colour = svdlut.cie94(y, t, CIE94_WEIGHT, dy=dy, accumulate=True)
        return {"mse": loss, "cie94": colour, "dy": dy}
    if kind == "train":
        x, t, dy, gen = state["x"], state["target"], state["dy"], state["gen"]
        p = gen.forward(x, training=True, seed=state["dropout_seed"])
        y = svdlut.apply(x, p)
        loss = svdlut.mse(y, t, dy)
        colour = svdlut.cie94(y, t, CIE94_WEIGHT, dy=dy, accumulate=True)
        g = svdlut.backward(x, p, dy, want=tuple("d" + n for n in svdlut.PARAM_NAMES))
        dw = gen.backward({n: g["d" + n] for n in svdlut.PARAM_NAMES})
        return {"params": p, "y": y, "mse": loss, "cie94": colour, "dparams": g, "dweights": dw}
    return svdlut.lut3d_apply(state["x"], state["lut"])


# ---------------------------------------------------------------- what one pass cannot do without

def _param_bytes(K, Dsx, Dsy):
    return 4 * (9 * RANK * (2 * DT + 1) + 12 + K * (Dsx * Dsy + DSC * (Dsx + Dsy) + 4))


APPLY_FLOPS = 3 * 3 * 9 + 3 * 3 * 5 + 3 * 6  # three pairs, three slices, cells; per pixel
GEN_MACS = sum(GEN_CHANNELS[i] * GEN_CHANNELS[i + 1] * 9 * (GEN_THUMB >> (i + 1)) ** 2 for i in range(5))


def _thumb_bytes(H, W):
    """Bytes of one frame that its 256 x 256 bilinear thumbnail reads (32-byte sectors)."""
    rows = min(H, 2 * GEN_THUMB)
    return 3 * rows * min(4 * W, 32 * 2 * GEN_THUMB)


def work(case):
    kind = case["kind"]
    if kind == "ragged":
        sizes = _ragged_sizes(case)
        px, es = sum(w * h for w, h in sizes), 4 if case["fmt"] == "f32" else 1
        return {"bytes": 6 * es * px + sum(_param_bytes(*_grid_dims("eighth", h, w)) for w, h in sizes),
                "flops": APPLY_FLOPS * px}
    B, H, W = case["B"], case["H"], case["W"]
    px = B * H * W
    if kind == "apply":
        fmt = case["fmt"]
        e_in = 4 if fmt == "f32" else (2 if fmt.startswith("u16") else 1)
        e_out = 4 if OUT_FORMAT.get(fmt, fmt) == "f32" else 1
        return {"bytes": 3 * (e_in + e_out) * px + B * _param_bytes(*_grid_dims(case["grids"], H, W)),
                "flops": APPLY_FLOPS * px}
    if kind == "backward":
        return {"bytes": 36 * px + 2 * B * _param_bytes(*_grid_dims(case["grids"], H, W)), "flops": 3 * APPLY_FLOPS * px}
    if kind == "loss":
        return {"bytes": 36 * px, "flops": 200 * px}
    if kind == "lut3d":
        return {"bytes": 24 * px + 12 * B * case["D"] ** 3, "flops": 60 * px}
    K = case["K"]
    weights = 4 * sum(math.prod(s) for _, s in _generator_shapes(K))
    params = B * _param_bytes(K, DSC, DSC)
    if kind == "generate":
        return {"bytes": B * _thumb_bytes(H, W) + weights + params, "flops": 2 * B * GEN_MACS}
    # x and target in, y, the factors, their gradients and the weights' gradient out
    return {"bytes": 36 * px + 2 * weights + 2 * params, "flops": 6 * B * GEN_MACS + (4 * APPLY_FLOPS + 200) * px}


# ---------------------------------------------------------------- the same in 64 bits

def _cell(u, D):
    """Cell index and offset of coordinates u = p (D - 1): on a vertex either neighbour gives the same value."""
    i = torch.clamp(torch.round(u - 0.5), max=D - 2)
    return i.long(), u - i


def _axis(n, Ds):
    """Cells of n pixels on Ds vertices."""
    k = torch.arange(n, device="cuda")
    if n == 1:
        return torch.zeros(1, dtype=torch.long, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    i = torch.clamp(k * (Ds - 1) // (n - 1), max=Ds - 2)
    return i, (k * (Ds - 1) - i * (n - 1)).double() / (n - 1)


def _bilinear(table, i, j, a, b, n_j):
    """table [V, C] with row i * n_j + j, at cells (i, j) with offsets (a, b) -> [P, C]."""
    r = i * n_j + j
    t00, t01 = table.index_select(0, r), table.index_select(0, r + 1)
    t10, t11 = table.index_select(0, r + n_j), table.index_select(0, r + n_j + 1)
    a, b = a[:, None], b[:, None]
    return (t00 * (1 - a) + t10 * a) * (1 - b) + (t01 * (1 - a) + t11 * a) * b


def _transform64(x, p):
    """The transform of one image x [3,H,W] by the factors p (no batch axis), float64."""
    _, H, W = x.shape
    q = x.reshape(3, -1).clamp(0, 1)
    D, K = p["U"].shape[-2], p["g_xy"].shape[0]
    T = torch.einsum("cpir,cpr,cpjr->pijc", p["U"], p["S"], p["V"])
    y = p["lut_w"][:, 3][None]
    cells = [_cell(q[c] * (D - 1), D) for c in range(3)]
    for pr, (A, Bx) in enumerate(((0, 1), (0, 2), (1, 2))):
        (ia, da), (ib, db) = cells[A], cells[Bx]
        y = y + _bilinear(T[pr].reshape(D * D, 3) * p["lut_w"][:, pr], ia, ib, da, db, D)
    if K:
        Dsy, Dsx, Dsc = p["g_xy"].shape[1], p["g_xy"].shape[2], p["g_xc"].shape[2]
        iy, ey = (t[:, None].expand(H, W).reshape(-1) for t in _axis(H, Dsy))
        ix, ex = (t[None].expand(H, W).reshape(-1) for t in _axis(W, Dsx))
        cols = []
        for c in range(3):
            w = p["grid_w"][c::3]
            fxy, fxc, fyc = (torch.einsum("k,kij->ij", w[:, n], p[g][c::3]).reshape(-1, 1)
                             for n, g in enumerate(("g_xy", "g_xc", "g_yc")))
            jc, ec = _cell(q[c] * (Dsc - 1), Dsc)
            cols.append(_bilinear(fxy, iy, ix, ey, ex, Dsx) + _bilinear(fxc, ix, jc, ex, ec, Dsc)
                        + _bilinear(fyc, iy, jc, ey, ec, Dsc) + w[:, 3].sum())
        y = y + torch.cat(cols, 1)
    return y.t().reshape(3, H, W)


def _image_params(params, b):
    return {k: v[b].double() for k, v in params.items()}


def _forward64(x, params):
    return torch.stack([_transform64(x[b].double(), _image_params(params, b)) for b in range(x.shape[0])])


def _backward64(x, params, dy):
    out = {}
    for b in range(x.shape[0]):
        xb = x[b].double().requires_grad_()
        p = {k: v.requires_grad_() for k, v in _image_params(params, b).items()}
        names = list(p)
        g = torch.autograd.grad(_transform64(xb, p), [xb] + [p[n] for n in names], dy[b].double())
        # a clamped input passes no gradient
        g = (g[0] * ((xb >= 0) & (xb <= 1)),) + g[1:]
        for n, v in zip(["x"] + names, g):
            out.setdefault("d" + n, []).append(v.detach())
    return {k: torch.stack(v) for k, v in out.items()}


def _splitmix64(x):
    with np.errstate(over="ignore"):
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _generate64(weights, K, x, dropout_seed=None):
    p, o = {}, 0
    for n, s in _generator_shapes(K):
        p[n] = weights[o:o + math.prod(s)].reshape(s)
        o += math.prod(s)
    F = torch.nn.functional
    B = x.shape[0]
    a = torch.cat([F.interpolate(x[b:b + 1].double(), (GEN_THUMB, GEN_THUMB), mode="bilinear") for b in range(B)])
    for i in range(5):
        cols = F.unfold(a, 3, padding=1, stride=2)  # [B, 9 Cin, P]
        side = a.shape[-1] // 2
        w = p[f"conv{i}.w"]
        z = (torch.matmul(w.reshape(w.shape[0], -1), cols) + p[f"conv{i}.b"][:, None]).reshape(B, -1, side, side)
        a = F.leaky_relu(z, 0.2)
        if i < 4:
            m, v = a.mean((2, 3), keepdim=True), a.var((2, 3), unbiased=False, keepdim=True)
            a = (a - m) / torch.sqrt(v + 1e-5) * p[f"in{i}.g"][:, None, None] + p[f"in{i}.b"][:, None, None]
    if dropout_seed is not None:
        e = (np.uint64(dropout_seed) << np.uint64(32)) + np.arange(B * 64 * 64, dtype=np.uint64)
        keep = (_splitmix64(e) >> np.uint64(63)) == 0
        a = a * torch.as_tensor(keep * 2.0, device="cuda").reshape(B, 64, 8, 8)
    rho = F.avg_pool2d(a, 4).reshape(B, 256)
    hs, hsw, ht, htw = ((rho @ p[f"h{h}.w1"].t() + p[f"h{h}.b1"]) @ p[f"h{h}.w2"].t() + p[f"h{h}.b2"]
                        for h in ("s", "sw", "t", "tw"))
    g, nu, ns = hs.reshape(B, K, 3, DSC, DSC), 9 * DT * RANK, 9 * RANK
    return {"U": ht[:, :nu].reshape(B, 3, 3, DT, RANK), "S": ht[:, nu:nu + ns].reshape(B, 3, 3, RANK),
            "V": ht[:, nu + ns:].reshape(B, 3, 3, DT, RANK), "lut_w": htw.reshape(B, 3, 4), "g_xy": g[:, :, 0],
            "g_xc": g[:, :, 1], "g_yc": g[:, :, 2], "grid_w": hsw.reshape(B, K, 4)}


def _white(x, y):
    return np.array([x / y, 1.0, (1.0 - x - y) / y])


def _lab(v):
    """CIELAB (D65) of sRGB images [B,3,H,W]."""
    prim = np.stack([_white(*c) for c in ((0.64, 0.33), (0.30, 0.60), (0.15, 0.06))], 1)
    white = _white(0.3127, 0.3290)
    m = torch.as_tensor(prim * np.linalg.solve(prim, white) / white[:, None], device="cuda")
    lin = torch.where(v <= 0.04045, v / 12.92, ((v.clamp(min=0.04045) + 0.055) / 1.055) ** 2.4)
    t = torch.einsum("ij,bjhw->bihw", m, lin)
    eps, kappa = 216.0 / 24389.0, 24389.0 / 27.0
    f = torch.where(t > eps, t.clamp(min=eps) ** (1.0 / 3.0), (kappa * t + 16.0) / 116.0)
    return 116.0 * f[:, 1] - 16.0, 500.0 * (f[:, 0] - f[:, 1]), 200.0 * (f[:, 1] - f[:, 2])


def _cie94(y, target):
    (l1, a1, b1), (l2, a2, b2) = _lab(target), _lab(y)
    c1, c2 = torch.sqrt(a1 * a1 + b1 * b1), torch.sqrt(a2 * a2 + b2 * b2)
    dl, dc, da, db = l1 - l2, c1 - c2, a1 - a2, b1 - b2
    dh2 = (da * da + db * db - dc * dc).clamp(min=0)
    return torch.sqrt(dl * dl + (dc / (1 + 0.045 * c1)) ** 2 + dh2 / (1 + 0.015 * c1) ** 2).mean()


def _loss64(y, target):
    """mse, cie94 and the gradient of mse + 0.005 cie94."""
    y = y.detach().requires_grad_()
    mse, colour = ((y - target) ** 2).mean(), _cie94(y, target)
    (dy,) = torch.autograd.grad(mse + CIE94_WEIGHT * colour, y)
    return mse.detach(), colour.detach(), dy


def _lut3d64(x, lut):
    D = lut.shape[-1]
    out = []
    for b in range(x.shape[0]):
        q = x[b].double().reshape(3, -1).clamp(0, 1) * (D - 1)
        i = torch.clamp(torch.floor(q), max=D - 2).long()
        d = q - i
        table = lut[b].double().reshape(3, -1).t().contiguous()
        y = 0
        for k in range(8):
            o = [(k >> 2) & 1, (k >> 1) & 1, k & 1]
            w = math.prod((d[c] if o[c] else 1 - d[c]) for c in range(3))
            y = y + w[:, None] * table.index_select(0, ((i[0] + o[0]) * D + i[1] + o[1]) * D + i[2] + o[2])
        out.append(y.t().reshape(x[b].shape))
    return torch.stack(out)


def exact(case, seed):
    kind = case["kind"]
    if case.get("fmt", "f32") not in ("f32", "u16"):
        return None  # 8-bit results are compared as bytes
    s = prepare(case, seed)
    if kind == "apply":
        if case["fmt"] == "u16":
            return _forward64(s["x"].to(torch.int32).double() / 65535.0, s["params"])
        return _forward64(s["x"], s["params"])
    if kind == "ragged":
        return [_transform64(x.double(), {k: v.double() for k, v in p.items()}) for x, p in zip(s["xs"], s["params"])]
    if kind == "backward":
        return _backward64(s["x"], s["params"], s["dy"])
    if kind == "generate":
        return _generate64(s["gen"].weights.double(), case["K"], s["x"])
    if kind == "loss":
        mse, colour, dy = _loss64(s["y"].double(), s["target"].double())
        return {"mse": mse, "cie94": colour, "dy": dy}
    if kind == "train":
        p = _generate64(s["gen"].weights.double(), case["K"], s["x"], s["dropout_seed"])
        y = _forward64(s["x"], p)
        mse, colour, dy = _loss64(y, s["target"].double())
        g = _backward64(s["x"], p, dy)
        # The early layers' weight gradients follow the signs that the LeakyReLUs of a bfloat16 network take: those of
        # a 64-bit network are another function's.
        return {"params": p, "y": y, "mse": mse, "cie94": colour,
                "dparams": {"d" + n: g["d" + n] for n in p}, "dweights": None}
    return _lut3d64(s["x"], s["lut"])
