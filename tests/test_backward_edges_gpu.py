"""Adjoint at the edges of its kernels' tiles, against the FP64 oracle.

Tolerances as tests/test_backward_gpu.py: FP32 sums of O(1) terms, parameter
gradients ||d - ref|| <= 1e-4 ||ref|| and max-abs <= 1e-3 max|ref|.
"""
import numpy as np
import pytest

import oracle
import svdlut_inputs as si

pytestmark = pytest.mark.gpu

NAMES = ("U", "S", "V", "lut_w", "g_xy", "g_xc", "g_yc", "grid_w")


def check(x, p, dy, d):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    g = sv.backward(torch.from_numpy(x).cuda(), sv.to_device(p), torch.from_numpy(dy).cuda(),
                    want=tuple("d" + n for n in NAMES))
    torch.cuda.synchronize()
    ref = oracle.backward(d, p, x, dy)
    for n in NAMES:
        a, r = g["d" + n].cpu().numpy().astype(np.float64), ref["d" + n]
        if r.size == 0:
            continue
        assert np.linalg.norm(a - r) <= 1e-4 * max(np.linalg.norm(r), 1e-30) + 1e-6, n
        assert np.abs(a - r).max() <= 1e-3 * np.abs(r).max() + 1e-6, n


# (H, W, grid dims): strips of 128 columns with 1, 127, 128 and 129 columns, a
# row group without rows, x-cells of 1, 2, 3 and 40 pixels and narrower than a
# pixel (the two ways that the xy sums are spread), y-cells of one row, more
# than 32 x vertices in a strip, the fewest and the most intensity vertices
@pytest.mark.parametrize("H,W,Dsx,Dsy,Dsc", [
    (3, 129, 129, 3, 2), (16, 127, 64, 16, 5), (17, 128, 43, 5, 2), (33, 257, 7, 33, 16), (40, 20, 31, 9, 17),
    (81, 300, 38, 11, 33), (18, 140, 9, 7, 64), (160, 96, 2, 2, 24)])
def test_grid_gradients_at_tile_edges(H, W, Dsx, Dsy, Dsc):
    d = si.Dims(9, 3, 5, Dsx, Dsy, Dsc)
    x, p = si.make_batch(700 + H + W, 2, H, W, d)
    check(x, p, si.make_upstream(701 + H, x.shape), d)


# (H, W, D_t, image): 64-column strips with 1, 63, 64 and 65 columns, shares
# without rows, one LUT cell and the largest table; every lane in one cell,
# every lane in its own, a few cells per warp, and runs that end a few lanes at
# a time (the queue)
@pytest.mark.parametrize("H,W,D,mode", [
    (1, 1, 2, "noise"), (2, 63, 33, "noise"), (5, 64, 33, "constant"), (3, 65, 17, "smooth"), (40, 130, 33, "noise"),
    (70, 97, 33, "dither"), (64, 64, 2, "noise"), (37, 200, 33, "smooth")])
def test_lut_gradients_at_strip_and_queue_edges(H, W, D, mode):
    d = si.Dims(D, min(D, 8), 3, 2, 2, 5)
    x, p = si.make_batch(720 + H + W, 2, H, W, d, mode=mode if mode in ("noise", "smooth") else "smooth")
    if mode == "constant":
        x[...] = np.float32(0.3125 + 1 / 64)
    if mode == "dither":  # flat areas whose pixels fall in a few neighbouring cells
        x = np.clip(0.4 + np.random.default_rng(722).normal(0, 0.02, x.shape), 0, 1).astype(np.float32)
    dy = si.make_upstream(721 + H, x.shape)
    check(x, p, dy, d)


def test_lut_gradients_are_bitwise_repeatable():
    import torch
    import paper_2508_16121_gb300 as sv
    H, W = 150, 333
    d = si.spatial_dims(H, W)
    x, p = si.make_batch(740, 2, H, W, d)
    xt, pt = torch.from_numpy(x).cuda(), sv.to_device(p)
    dy = torch.from_numpy(si.make_upstream(741, x.shape)).cuda()
    first = sv.backward(xt, pt, dy)
    for _ in range(3):
        again = sv.backward(xt, pt, dy)
        for k in first:
            assert torch.equal(first[k], again[k]), k


# shares of the LUT pass that end inside images, hold several whole ones, are
# one row, or are fewer than the SMs (batch, H, W)
@pytest.mark.parametrize("B,H,W", [(7, 45, 70), (160, 3, 65), (3, 1, 1), (64, 40, 64), (5, 171, 129)])
def test_lut_shares_across_images(B, H, W):
    d = si.Dims(17, 4, 3, 3, 3, 5)
    x, p = si.make_batch(900 + B, B, H, W, d)
    check(x, p, si.make_upstream(901 + B, x.shape), d)
