"""The loss kernels at the edges of their access widths: planes that are not
a multiple of four pixels, arrays off a 16-byte boundary, remainders, several
turns per thread."""
import numpy as np
import pytest

from oracle import cie94 as ocie

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    import torch
    import paper_2508_16121_gb300 as svdlut
    from paper_2508_16121_gb300 import build
    build.build()
    assert torch.cuda.is_available()
    return svdlut


def _at(a, off):
    """The array on the GPU, off floats past an allocation's start."""
    import torch
    buf = torch.empty(a.size + off, dtype=torch.float32, device="cuda")
    v = buf[off:].view(a.shape)
    v.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return v


@pytest.mark.parametrize("off", [(0, 0, 0), (1, 0, 0), (0, 2, 0), (0, 0, 3)])
@pytest.mark.parametrize("B,H,W", [(1, 1, 4), (3, 5, 7), (2, 2, 2), (5, 64, 66), (3, 301, 1031), (9, 512, 260)])
def test_cie94_and_mse(sv, B, H, W, off):
    import torch
    rng = np.random.default_rng(B * 1000 + W)
    t = rng.uniform(0, 1, (B, 3, H, W)).astype(np.float32)
    y = np.clip(t + rng.normal(0, 0.05, t.shape), -0.2, 1.2).astype(np.float32)
    yt, tt = _at(y, off[0]), _at(t, off[1])
    dy = _at(np.zeros_like(y), off[2])
    y64, t64 = y.astype(np.float64), t.astype(np.float64)

    loss = float(sv.mse(yt, tt, dy))
    # fp32 sums of at most a few hundred terms per thread, then per block
    assert loss == pytest.approx(((y64 - t64) ** 2).mean(), rel=1e-5)
    g = 2 * (y64 - t64) / y.size
    # one subtraction and one product in FP32: 2 roundings of values <= 1.4 each
    assert np.abs(dy.cpu().numpy() - g).max() <= 4 * 2.0 ** -24 * 2 * 1.4 / y.size

    w = 0.01
    colour = float(sv.cie94(yt, tt, weight=w, dy=dy, accumulate=True))
    assert colour == pytest.approx(ocie.cie94_loss(y64, t64), rel=1e-5)
    gref = w * ocie.cie94_grad(y64, t64)
    assert np.abs(dy.cpu().numpy() - g - gref).max() <= 1e-3 * np.abs(gref).max()
    assert float(sv.cie94(yt, tt)) == colour  # without a gradient
    assert torch.equal(yt.cpu(), torch.from_numpy(y))
