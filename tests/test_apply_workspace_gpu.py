"""svdlut_apply_ws and svdlut_apply_batched take their per-image tables from the
workspace for small calls too, eager and replayed from a CUDA graph: a call with
a workspace is written for the GPU's time, whatever the caller's own costs.  The
results are svdlut_apply's, bit for bit."""
import numpy as np
import pytest

import oracle
import svdlut_inputs as si

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 64, 64), (1, 256, 250), (4, 64, 64), (15, 48, 52)]


def _data(B, H, W):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import build
    build.build()
    d = si.spatial_dims(H, W)
    x, p = si.make_batch(1500 + B + H, B, H, W, d)
    xt, pt = torch.from_numpy(x).cuda(), sv.to_device(p)
    return torch, sv, xt, pt, oracle.forward(d, p, x)


@pytest.mark.parametrize("B,H,W", SHAPES)
def test_small_calls_take_the_tables(B, H, W):
    torch, sv, xt, pt, ref = _data(B, H, W)
    plain = sv.apply(xt, pt, workspace=False)
    assert np.abs(plain.cpu().numpy() - ref).max() <= 2e-5
    need = sv._lib.load().svdlut_apply_workspace_size(sv.dims_of(pt), B)
    ws = torch.full((need,), 0xAB, dtype=torch.uint8, device="cuda")
    assert torch.equal(sv.apply(xt, pt, workspace=ws), plain)
    per = need // B
    for b in range(B):  # the cell table of every image is there
        assert not bool((ws[b * per:b * per + 1024] == 0xAB).all()), b
    one = [{n: t[b].contiguous() for n, t in pt.items()} for b in range(B)]
    batch = sv.Batch([xt[b].contiguous() for b in range(B)], one)
    batch.ws.fill_(0xAB)
    for b, y in enumerate(batch.run()):
        assert torch.equal(y, plain[b])
    assert not bool((batch.ws[256:1280] == 0xAB).all())


# the default of the Python call, from the eager route to the captured one
@pytest.mark.parametrize("B,H,W", SHAPES)
@pytest.mark.parametrize("explicit", [False, True])
def test_captured_calls_take_the_tables(B, H, W, explicit):
    torch, sv, xt, pt, ref = _data(B, H, W)
    eager = sv.apply(xt, pt)
    assert np.abs(eager.cpu().numpy() - ref).max() <= 2e-5
    y = torch.full_like(xt, float("nan"))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    taken = []
    real = sv._stream_workspace
    sv._stream_workspace = lambda *a: taken.append(a[1]) or real(*a)
    try:
        with torch.cuda.graph(g, stream=s):
            sv.apply(xt, pt, out=y, stream=s if explicit else None)
    finally:
        sv._stream_workspace = real
    assert taken == [sv._lib.load().svdlut_apply_workspace_size(sv.dims_of(pt), B)]
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, eager)
