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
