"""The adjoint with so many y vertices per image row that only blocks of few
rows fit its kernels, against the FP64 oracle (tolerances as
tests/test_backward_gpu.py: FP32 sums of O(1) terms, ||d - ref|| <= 1e-4 ||ref||
and max-abs <= 1e-3 max|ref|); dx, which no plan of these changes, as asked for
alone."""
import numpy as np
import pytest

import oracle
import svdlut_inputs as si

pytestmark = pytest.mark.gpu

NAMES = ("U", "S", "V", "lut_w", "g_xy", "g_xc", "g_yc", "grid_w")


# 8 vertices per row at Dsc = 64 (the tallest block that fits: 11 rows), 7.5 (13
# of 14), 12.5 at 48 (10), and 31 and 16 per row in blocks of whole bands
@pytest.mark.parametrize("B,H,W,d", [
    (2, 16, 256, si.Dims(17, 8, 6, 17, 129, 64)), (1, 40, 100, si.Dims(9, 3, 5, 5, 300, 64)),
    (1, 30, 70, si.Dims(9, 3, 4, 3, 600, 48)), (2, 18, 100, si.Dims(9, 3, 5, 5, 559, 17)),
    (2, 20, 130, si.Dims(9, 3, 5, 9, 321, 33))])
def test_dense_y_vertices(B, H, W, d):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    x, p = si.make_batch(1300 + H + W, B, H, W, d)
    dy = si.make_upstream(1301 + H, x.shape)
    xt, pt, gt = torch.from_numpy(x).cuda(), sv.to_device(p), torch.from_numpy(dy).cuda()
    g = sv.backward(xt, pt, gt)
    again = sv.backward(xt, pt, gt)
    torch.cuda.synchronize()
    ref = oracle.backward(d, p, x, dy)
    assert torch.equal(sv.backward(xt, pt, gt, want=("dx",))["dx"], g["dx"])
    for n in tuple("d" + n for n in NAMES):
        a, r = g[n].cpu().numpy().astype(np.float64), ref[n]
        assert np.linalg.norm(a - r) <= 1e-4 * max(np.linalg.norm(r), 1e-30) + 1e-6, n
        assert np.abs(a - r).max() <= 1e-3 * np.abs(r).max() + 1e-6, n
        assert torch.equal(g[n], again[n]), n
