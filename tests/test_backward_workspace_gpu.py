"""The adjoint with as little workspace as svdlut_backward_noalloc's scratch
leaves it, against the same call with the workspace that it asks for.

Both plans sum the same terms in another order: FP32 sums of O(1) terms, the
adjoint tests' tolerances."""
import ctypes

import numpy as np
import pytest

import svdlut_inputs as si

pytestmark = pytest.mark.gpu

NAMES = ("U", "S", "V", "lut_w", "g_xy", "g_xc", "g_yc", "grid_w")


# batches whose fastest plan is beyond the scratch: 51 LUT CTAs of three images
# each, 77 of two, 31 of five
@pytest.mark.parametrize("B", [153, 154, 155])
def test_plan_within_the_fixed_scratch(B):
    import torch
    import paper_2508_16121_gb300 as sv
    from paper_2508_16121_gb300 import _lib
    lib = _lib.load(build_if_missing=True)
    H, W = 40, 72
    d = si.Dims(33, 8, 8, 17, 17, 17)
    x, p = si.make_batch(1200 + B, B, H, W, d)
    xt, pt = torch.from_numpy(x).cuda(), sv.to_device(p)
    dy = torch.from_numpy(si.make_upstream(1201 + B, x.shape)).cuda()
    ref = sv.backward(xt, pt, dy)
    dims = sv.dims_of(pt)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert lib.svdlut_backward_workspace_size(dims, B, H, W) > 32 << 20
    outs = {"d" + n: torch.full_like(pt[n], float("nan")) for n in NAMES}
    g = _lib.Grads(**{k: v.data_ptr() for k, v in outs.items()})
    dx = torch.full_like(xt, float("nan"))
    st = lib.svdlut_backward_noalloc(dims, sv._param_struct(pt, B, dims), B, H, W, xt.data_ptr(), dy.data_ptr(),
                                     dx.data_ptr(), g, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0, lib.svdlut_last_error()
    torch.cuda.synchronize()
    assert torch.equal(dx, ref["dx"])
    for k, v in outs.items():
        a, r = v.cpu().numpy().astype(np.float64), ref[k].cpu().numpy().astype(np.float64)
        assert np.linalg.norm(a - r) <= 1e-4 * np.linalg.norm(r) + 1e-6, k
        assert np.abs(a - r).max() <= 1e-3 * np.abs(r).max() + 1e-6, k
