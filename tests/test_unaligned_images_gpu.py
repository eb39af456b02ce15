"""Float images whose rows start at every offset from a 16-byte boundary: the
same bits whatever the offset of the arrays, for transform and adjoint, and
within the oracle's tolerance (max-abs 2e-5)."""
import numpy as np
import pytest

import oracle
import svdlut_inputs as si

pytestmark = pytest.mark.gpu


def _at(a, off):
    """Array a on the GPU, off floats past an allocation's start."""
    import torch
    buf = torch.zeros(a.size + off + 4, dtype=torch.float32, device="cuda")
    v = buf[off:off + a.size].view(a.shape)
    v.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return buf, v


# odd, even and fourfold widths, and plane sizes of every remainder; a width
# below a lane's four pixels, lanes that end inside a strip
@pytest.mark.parametrize("B,H,W", [(1, 9, 131), (2, 7, 130), (1, 6, 133), (1, 5, 128), (2, 3, 3), (1, 33, 258), (17, 180, 181)])
def test_every_offset_gives_the_same_bits(B, H, W):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    d = si.Dims(33, 8, 6, 17, 17, 17) if B > 2 else si.spatial_dims(H, W)
    x, p = si.make_batch(5200 + W, B, H, W, d)
    pd = sv.to_device(p)
    dy = si.make_upstream(5201 + W, x.shape)
    ref = None
    for off in range(4):
        _, xt = _at(x, off)
        buf, y = _at(np.zeros_like(x), (off + 1) % 4)
        sv.apply(xt, pd, out=y)
        got = {"y": y.clone(), **sv.backward(xt, pd, _at(dy, (off + 2) % 4)[1])}
        # nothing written outside the result
        assert float(buf[:(off + 1) % 4].abs().sum()) == 0.0 and float(buf[(off + 1) % 4 + x.size:].abs().sum()) == 0.0
        if ref is None:
            ref = got
            assert np.abs(y.cpu().numpy().astype(np.float64) - oracle.forward(d, p, x)).max() <= 2e-5
        for n in ref:
            assert torch.equal(got[n], ref[n]), (n, off)
