"""The ways to an image's tables (the rank-8 build in every CTA, the general
build, the workspace's precomputed tables or its folded grids alone) against
the FP64 oracle (max-abs 2e-5) and, bit for bit, against one another."""
import numpy as np
import pytest

import oracle
import svdlut_inputs as si

pytestmark = pytest.mark.gpu

TOL = 2e-5


def _unaligned(t):
    import torch
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = buf[1:].view(t.shape)
    v.copy_(t)
    return v


# D_t from the smallest with rank 8 to the largest (7 to 32 cells per axis: fewer rows than
# a warp, segments of unequal length), no grids, fewer grids than channels,
# fast and general rows, a slope-form xc slice (too small for the factors),
# rank 7 (general build)
@pytest.mark.parametrize("d,B,H,W", [
    (si.Dims(8, 8, 1, 2, 2, 2), 1, 5, 9), (si.Dims(9, 8, 0, 2, 2, 2), 2, 40, 131), (si.Dims(16, 8, 2, 5, 4, 9), 1, 33, 260),
    (si.Dims(32, 8, 8, 17, 17, 17), 3, 70, 129), (si.Dims(33, 8, 6, 17, 17, 17), 2, 257, 300),
    (si.Dims(33, 8, 8, 90, 9, 17), 1, 64, 181), (si.Dims(33, 8, 4, 6, 6, 40), 1, 50, 200), (si.Dims(17, 7, 5, 6, 6, 9), 1, 50, 200),
    (si.spatial_dims(853, 400), 1, 853, 400),
    # more pixels than one launch's worth: tables from prep_kernel, and from 16 images on the folded grids
    (si.spatial_dims(700, 757), 1, 700, 757), (si.Dims(33, 8, 6, 17, 17, 17), 15, 200, 180),
    (si.Dims(33, 8, 6, 17, 17, 17), 16, 200, 165), (si.Dims(17, 8, 4, 9, 5, 9), 20, 180, 148),
    (si.Dims(33, 8, 4, 17, 17, 12), 17, 190, 166)])
def test_every_way_gives_the_same_bits(d, B, H, W):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    x, p = si.make_batch(4100 + H + W, B, H, W, d)
    xt, pd = torch.from_numpy(x).cuda(), sv.to_device(p)
    y = sv.apply(xt, pd)
    assert np.abs(y.cpu().numpy().astype(np.float64) - oracle.forward(d, p, x)).max() <= TOL
    assert torch.equal(sv.apply(xt, pd, workspace=False), y)
    assert torch.equal(sv.apply(xt, pd, ctas=7), y)
    assert torch.equal(sv.apply(xt, {n: _unaligned(t) for n, t in pd.items()}, workspace=False), y)
    one = [{n: t[b].contiguous() for n, t in pd.items()} for b in range(B)]
    for out in sv.Batch([xt[b] for b in range(B)], one).run(), sv.Batch([xt[b] for b in range(B)], one, tables=False).run():
        for b in range(B):
            assert torch.equal(out[b], y[b])
