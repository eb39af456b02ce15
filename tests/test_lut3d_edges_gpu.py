"""The 3D LUT's gathers from shared memory and through L1: the same values on
both sides of the rule, for one channel and three channels per CTA, remainders
of the vector width, shares that end inside images, and in place."""
import numpy as np
import pytest

import oracle
import svdlut_inputs as si

pytestmark = pytest.mark.gpu

TOL = 1e-5  # as tests/test_lut3d_gpu.py


# 512 x 512 = 2^18 pixels: the fewest that go through shared memory; 25: the
# largest table whose three channels fit, 26: the smallest that does not
@pytest.mark.parametrize("B,H,W,D", [(1, 512, 512, 33), (1, 511, 513, 33), (2, 517, 519, 33), (3, 600, 521, 25), (1, 640, 480, 26),
                                     (2, 512, 514, 2), (1, 512, 513, 17), (5, 700, 400, 33)])
def test_shared_gathers(B, H, W, D):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    rng = np.random.default_rng(3000 + W + D)
    lut = np.stack([si.make_lut3d(rng, D, "photo") for _ in range(B)]).astype(np.float32)
    x = np.stack([si.make_image(rng, H, W) for _ in range(B)]).astype(np.float32)
    x[:, :, ::7, ::5] = rng.uniform(-0.5, 1.5, x[:, :, ::7, ::5].shape)
    xt, lt = torch.from_numpy(x).cuda(), torch.from_numpy(lut).cuda()
    y = sv.lut3d_apply(xt, lt)
    assert np.abs(y.cpu().numpy() - oracle.lut3d_apply(lut, x)).max() <= TOL
    # rows of the images, few enough for the other kernel: the same bits
    part = xt[:, :, :100].contiguous()
    assert torch.equal(sv.lut3d_apply(part, lt), y[:, :, :100])
    # off a 16-byte boundary, and in place
    buf = torch.empty(x.size + 1, device="cuda")
    xu = buf[1:].view(x.shape)
    xu.copy_(xt)
    assert torch.equal(sv.lut3d_apply(xu, lt), y)
    assert torch.equal(sv.lut3d_apply(xu, lt, out=xu), y)
