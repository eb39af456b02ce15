"""The adjoint's launch plans (no GPU needed): a program that includes the
adjoint's source prints them for the sizes given, for a GPU of 152 SMs with 227
KB of shared memory per CTA."""
import math
import subprocess

import pytest

from paper_2508_16121_gb300 import build

SMS = 152
SCRATCH = 32 << 20  # svdlut_backward_noalloc's

PROGRAM = r'''
#include "svdlut_backward.cu"
#include <cstdio>
#include <cstring>
// "plan": a line "D_t rank K Dsx Dsy Dsc B H W" each -> two of "status bytes
// LUT-CTAs block-rows row-groups", without a limit and within the scratch
static void plans()
{
    svdlut_dims d;
    int B, H, W;
    while (scanf("%d%d%d%d%d%d%d%d%d", &d.D_t, &d.rank, &d.K, &d.Dsx, &d.Dsy, &d.Dsc, &B, &H, &W) == 9) {
        for (size_t limit : {size_t(SIZE_MAX), kNoAllocScratchBytes}) {
            BwdPlan p{};
            const int st = plan_backward(&d, B, H, W, 152, 227 * 1024, limit, &p);
            printf("%d %zu %d %d %d ", st, p.total, p.G, p.gp.BH, p.gp.groups);
        }
        printf("\n");
    }
}
// "slots": a line "G B units" each -> 1 if the parts of G shares of B images of
// so many units have a slot each below lut_slot_count, in order, and lut_slots
// names every image's, no other's among them
static void slots()
{
    int G, B;
    long long per;
    while (scanf("%d%d%lld", &G, &B, &per) == 3) {
        const int seg = lut_segment(G, B), count = static_cast<int>(lut_slot_count(G, B));
        int prev = -1, good = 1;
            std::vector<int> first(B, -1), last(B, -1);
        for (int g = 0; g < G; ++g) {
            const long long c1 = lut_share(per * B, G, g + 1);
            for (long long c = lut_share(per * B, G, g); c < c1;) {
                const int b = static_cast<int>(c / per), s = lut_slot(g, b, seg);
                good &= s > prev && s < count && (first[b] < 0 || s == last[b] + 1);
                prev = s;
                if (first[b] < 0) first[b] = s;
                last[b] = s;
                c = std::min(c1, per * (b + 1));
            }
        }
        for (int b = 0; b < B; ++b) {
            int s0, s1;
            lut_slots(per, B, G, seg, b, s0, s1);
            good &= s0 == first[b] && s1 == last[b] + 1;
        }
        printf("%d\n", good);
    }
}
int main(int argc, char **argv)
{
    if (argc == 2 && !strcmp(argv[1], "plan")) plans();
    if (argc == 2 && !strcmp(argv[1], "slots")) slots();
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("plan")
    lib = build.build()
    src, exe = tmp / "plan.cu", tmp / "plan"
    src.write_text(PROGRAM)
    r = subprocess.run([build.nvcc()] + build.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I" + build.INCLUDE, "-I" + build.CSRC, str(src), lib, "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(what, lines):
        text = "\n".join(" ".join(str(v) for v in ln) for ln in lines)
        out = subprocess.run([str(exe), what], input=text, capture_output=True, text=True, timeout=300)
        assert out.returncode == 0, out.stderr
        return [[int(v) for v in ln.split()] for ln in out.stdout.splitlines()]

    return run


def test_large_batches_keep_the_gpu_full(program):
    """A workspace that the caller allocates does not limit the LUT pass, and
    the fixed scratch leaves each CTA few images (here it holds up to 154)."""
    batches = list(range(100, 201))
    for B, p in zip(batches, program("plan", [(33, 8, 8, 17, 17, 17, B, 256, 256) for B in batches])):
        assert p[0] == 0 and p[2] >= SMS - 8, (B, p)
        assert p[5] == 0 and (p[6] <= SCRATCH or B > 154), (B, p)
        if p[6] <= SCRATCH:
            assert -(-B // p[7]) <= 3, (B, p)
    frames = list(range(1, 30))
    for B, p in zip(frames, program("plan", [(33, 8, 8, 240, 135, 17, B, 1080, 1920) for B in frames])):
        assert p[0] == 0 and p[2] >= SMS - 8, (B, p)


def test_every_part_has_its_slot(program):
    cases = [(G, B, per) for G in (1, 2, 6, 7, 77, 150, 151, 152) for B in (1, 2, 3, 8, 64, 76, 77, 152, 154, 304)
             for per in (1, 5, 152, 1080) if G <= B * per]
    for c, (good,) in zip(cases, program("slots", cases)):
        assert good == 1, c


def _span(extent, n, ds):
    """Vertices that `extent` adjacent pixels of an axis of n touch, at most."""
    if n <= 1:
        return min(2, ds)
    return min(ds, math.ceil((extent - 1) * ((ds - 1) / (n - 1))) + 3)


def _taken(D, R, K, Dsx, Dsy, Dsc, B, H, W):
    """The densities that the adjoint takes: in some block of a band of the
    image, 16 warps' vertices of three channels within the shared memory."""
    nvx = _span(128, W, Dsx)
    for bands in range(1, max(1, -(-H // 16)) + 1):
        BH = -(-H // bands)
        ny = _span(-(-BH // 16), H, Dsy)
        if 4 * 16 * ((3 * (ny * nvx + (nvx + ny) * Dsc) + 3) // 4 * 4) + 256 <= 227 * 1024:
            return True
    return False


def test_dense_grids_are_taken(program):
    """Many y vertices per image row, up to the densest grids that the adjoint
    takes: every one of those has a plan whose blocks fit."""
    cases = [(17, 8, 6, 17, 129, 64, 1, 16, 256)]
    for Dsc in (2, 5, 9, 17, 24, 33, 48, 64):
        for H, W in ((1, 1), (3, 70), (16, 256), (20, 130), (37, 300), (200, 90)):
            for per_row in (1, 3, 6, 8, 12, 16, 24, 32, 48, 64):
                for Dsx in (2, 5, max(2, W // 8), max(2, W // 2)):
                    cases.append((9, 3, 4, Dsx, max(2, H * per_row), Dsc, 2, H, W))
    assert any(_taken(*c) for c in cases) and not all(_taken(*c) for c in cases)
    for c, p in zip(cases, program("plan", cases)):
        assert (p[0] == 0) == _taken(*c), (c, p)
