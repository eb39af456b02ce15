"""The 3D LUT of one large image, whose gathers come from shared memory, at the
smallest table and on both sides of the largest whose three channels fit a CTA
(25; 24 below it), with planes that are and are not a multiple of four pixels;
and batches of such images, which gather through L1: the oracle's values (max-abs
1e-5, as tests/test_lut3d_gpu.py) and, image by image, the same bits."""
import numpy as np
import pytest

import oracle
import svdlut_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W", [(520, 512), (511, 515)])
@pytest.mark.parametrize("D", [2, 3, 24, 25, 26])
def test_one_image_and_batches_give_the_same_bits(D, H, W):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    rng = np.random.default_rng(3300 + W + D)
    lut = np.stack([si.make_lut3d(rng, D, "photo") for _ in range(2)]).astype(np.float32)
    x = np.stack([si.make_image(rng, H, W) for _ in range(2)]).astype(np.float32)
    x[:, :, ::5, ::3] = rng.uniform(-0.5, 1.5, x[:, :, ::5, ::3].shape)
    x[:, 0, 0, :4] = (0.0, 1.0, np.nan, np.inf)
    xt, lt = torch.from_numpy(x).cuda(), torch.from_numpy(lut).cuda()
    both = sv.lut3d_apply(xt, lt)
    for b in range(2):
        one = sv.lut3d_apply(xt[b], lt[b])
        assert torch.equal(one, both[b])
        assert np.abs(one.cpu().numpy()[:, 1:] - oracle.lut3d_apply(lut[b:b + 1], x[b:b + 1])[0][:, 1:]).max() <= 1e-5
