"""The index-checked build (-DSVDLUT_CHECK_BOUNDS) in the instances that take
their tables, or the folded grids, from the workspace, which serve large frames
and large batches: no index out of range, no misaligned access or copy, and the
FP64 oracle's results.  Sizes by launch_tables's rule (csrc/apply_launch.cuh)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = r'''
import numpy as np, torch
import svdlut_inputs as si
import oracle
import paper_2508_16121_gb300 as sv
worst = 0.0

def close(y, ref):
    global worst
    worst = max(worst, float(np.abs(y.cpu().numpy() - ref).max()))

def unaligned(t):
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = buf[1:].view(t.shape)
    v.copy_(t)
    return v

# frames: all tables from the workspace, fast and general rows, aligned and unaligned images
for (B, H, W, d) in [(1, 720, 1280, si.spatial_dims(720, 1280)), (1, 700, 757, si.spatial_dims(700, 757)),
                     (1, 700, 751, si.Dims(33, 8, 6, 17, 17, 12)), (2, 512, 600, si.Dims(17, 7, 5, 6, 6, 40))]:
    x, p = si.make_batch(5 + H + W, B, H, W, d)
    xt, pd = torch.from_numpy(x).cuda(), sv.to_device(p)
    ref = oracle.forward(d, p, x)
    close(sv.apply(xt, pd), ref)
    close(sv.apply(unaligned(xt), pd), ref)
    sv.apply((xt * 255).round().clamp(0, 255).to(torch.uint8), pd)
# many images: folded grids from the workspace, the cells from factors in the CTAs; and small ones, nothing
for (B, H, W, d) in [(17, 180, 180, si.Dims(33, 8, 6, 17, 17, 17)), (40, 128, 130, si.Dims(17, 8, 4, 9, 5, 9)),
                     (16, 20, 24, si.Dims(33, 8, 6, 17, 17, 17)), (64, 96, 100, si.Dims(33, 8, 6, 17, 17, 17))]:
    x, p = si.make_batch(6 + H + W, B, H, W, d)
    xt, pd = torch.from_numpy(x).cuda(), sv.to_device(p)
    ref = oracle.forward(d, p, x)
    close(sv.apply(xt, pd), ref)
    sv.apply((xt * 255).round().clamp(0, 255).to(torch.uint8), pd)
    one = [{n: t[b].contiguous() for n, t in pd.items()} for b in range(B)]
    for b, y in enumerate(sv.Batch([xt[b].contiguous() for b in range(B)], one).run()):
        close(y, ref[b])
    sv.backward(xt, pd, torch.from_numpy(si.make_upstream(7, x.shape)).cuda())
torch.cuda.synchronize()
rep = sv.check_report()
print("REPORT", rep, "WORST", worst)
assert rep is not None and rep["failures"] == 0, rep
assert worst <= 2e-5, worst
'''


def test_checked_build_of_the_table_instances(tmp_path):
    from paper_2508_16121_gb300 import build
    lib = str(tmp_path / "libsvdlut_checked.so")
    build.build(force=True, extra_flags=("-DSVDLUT_CHECK_BOUNDS",), out=lib)
    env = dict(os.environ, SVDLUT_LIB=lib)
    r = subprocess.run([sys.executable, "-c", CASES], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    print(r.stdout[-3000:], r.stderr[-4000:])
    assert r.returncode == 0
    assert "REPORT" in r.stdout
