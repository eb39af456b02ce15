// svdlut_backward: adjoint of the fused transform (FP32 images).
//
// The paper trains end to end through its slicing + LUT transform (Sec. 4.2)
// and prints no derivative; everything here is the exact derivative of the
// forward map of Eq. 10 / Supp. Eqs. 12-22.  Passes (all on the caller's
// stream, no atomics, every sum in a fixed order -> bitwise repeatable):
//   1. dx      : apply_kernel<IoF32, N, true> (slopes of the same cells).
//   2. lut     : lut_grad_kernel adds dy * bilinear weights to warp-private
//                tables G_p[i][j][c] (one LUT pair, all three output channels
//                per warp), then sums the warps of a CTA into a per-CTA
//                partial.
//   3. grid    : grid_grad_kernel sums the folded grid planes (xy, xc, yc per
//                output channel) over 128-px column blocks, in lane-private
//                bins.
//   4. reduce  : lut_finalize_kernel sums the CTA partials and contracts
//                through T = U diag(S) V^T (Eq. 9) to dU, dS, dV, dlut_w;
//                grid_reduce_kernel sums the block partials per vertex into dg_*
//                and per-CTA partials of dgrid_w, grid_wsum_kernel sums those.
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>
#include <cmath>
#include <cstdint>

#include "apply_kernel.cuh"
#include "apply_launch.cuh"

namespace svdlut {

// Fixed-order warp sum (butterfly); every lane gets the total.
__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct BwdArgs {
    const float *x, *dy;
    int B, H, W;
    int D, K, Dsx, Dsy, Dsc;
    float rW1, rH1;
    int strips;
    int vec;  // 16-byte loads allowed
    int seg;  // LUT pass: lut_segment
};

// ---------------------------------------------------------------------------
// LUT gradients: G^c_p[i][j] = sum_px dy_c * bilinear weight of vertex (i, j)
// at (x_alpha, x_beta) for pair p = (alpha, beta).
// The work is the sequence of (image, 64-column strip, row) triples; CTA g of G
// takes the g-th share of it (equal to within one row), one image's part of it
// after another, and row group g of the CTA the g-th share of a part.  Shares
// of the whole batch, not of an image: 64 images of 256 x 256 on 152 SMs take
// 152 CTAs, where whole CTAs per image left 24 SMs idle.
// Warp (pair q, group g) walks down the rows of its share; lane l takes
// columns l and l + 32 and keeps, per column, the twelve corner sums (four
// corners, three channels) of its current cell in registers: while the cell
// does not change it only accumulates.  Finished sums wait in the warp's queue
// (or, when most lanes finish at once, go straight on) until a batch of about
// 32 is there: equal cells are added up (match, rank tree), then one lane per
// cell adds its sums to the warp's own table [D][D][3], a corner at a time
// with a warp barrier between, so two cells never update one vertex in the
// same step.  The order of every sum is fixed: bitwise repeatable.
// Where a run ends a few lanes at a time (smooth content: neighbouring columns
// cross a cell border at different rows), the queue turns many nearly empty
// batches into a full one.  Tables of three floats per vertex (13 KB) leave
// room for 15 warps and their queues.  Noise, a new cell at every pixel, is
// bound by the shared-memory pipe (about 85 wavefronts a batch); smooth
// content by latency and issue slots, photos with pixel noise by the trees.
// Measured on 8 x 1920x1080, with lut_finalize_kernel: noise 534 us, smooth
// 310, half and half 413 (710 when each change of a lane's cell was scattered
// at once, from 12 warps with four floats per vertex).  Also tried, with whole
// CTAs per image, where the present way took 538, 287 and 429: one table
// of cells (48 bytes at one place, 66 wavefronts a batch) per pair, which its
// warps update in turns: 660, 440 and 563 us, the hand-over's latency; 12
// warps of this kernel: 580, 323, 460 us; the queue for every batch: 671,
// 282, 491 us.
// Output per part of CTA g and image b, in slot lut_slot(g, b): lut_part
// [slot][c][pair][D*D], sums_part[slot][c] (sum of dy_c).
// ---------------------------------------------------------------------------
constexpr int kLutGroups = 5, kLutWarps = 3 * kLutGroups;
constexpr int kLutThreads = kLutWarps * 32;
constexpr int kLutTileW = 64;   // columns of a strip: 32 lanes x 2
constexpr int kLutQueue = 32;   // queued sums of a warp
constexpr int kLutDirect = 14;  // lanes finishing at once from which the queue is passed by

// floats of one warp's queue, and of one table (rounded to 4: the queues follow)
constexpr int kLutQueueFloats = kLutQueue * 13;
__host__ __device__ inline int lut_table_floats(int D) { return (3 * D * D + 3) & ~3; }
__host__ __device__ inline size_t lut_grad_smem(int D)
{
    return sizeof(float) * (kLutWarps * (static_cast<size_t>(lut_table_floats(D)) + kLutQueueFloats) + 4 * kLutGroups);
}

// Shares of the LUT pass: work units [share(g), share(g + 1)) belong to CTA g.
__host__ __device__ inline long long lut_share(long long units, int G, int g) { return units * g / G; }
// The slot of CTA g's part of image b: a CTA's next image, and an image's next
// CTA, is the next slot.  Where a share ends with an image, both are next at
// once: with d = gcd(G, B) that is at every multiple of G / d shares (a segment)
// = B / d images, so G shares of B images have at most G + B - d parts.
__host__ __device__ inline int lut_segment(int G, int B)
{
    int a = G, b = B;
    while (b) {
        const int t = a % b;
        a = b;
        b = t;
    }
    return G / a;
}
__host__ __device__ inline int lut_slot(int g, int b, int seg) { return g + b - g / seg; }
inline size_t lut_slot_count(int G, int B) { return static_cast<size_t>(G) + B - G / lut_segment(G, B); }
// The slots of image b's parts, one per CTA that holds some of it.
__host__ __device__ inline void lut_slots(long long per_image, int B, int G, int seg, int b, int &s0, int &s1)
{
    const long long U = per_image * B;
    auto owner = [&](long long u) { return static_cast<int>(((u + 1) * G + U - 1) / U - 1); };
    s0 = lut_slot(owner(per_image * b), b, seg);
    s1 = lut_slot(owner(per_image * (b + 1) - 1), b, seg) + 1;
}

// Adds the 12 sums of lanes with equal keys (key < 0: none) into the lowest
// of them, by a tree over their ranks; returns whether this lane leads a key.
__device__ __forceinline__ bool merge_equal_keys(int key, float (&v)[12])
{
    const unsigned int full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned int me = 1u << lane, lower = me - 1u;
    const unsigned int grp = __match_any_sync(full, key >= 0 ? key : -1 - lane);
    unsigned int g = grp;  // members that still hold a partial sum
    while (__any_sync(full, (g & (g - 1u)) != 0u)) {
        const unsigned int above = g & ~(me | lower);
        const bool even = (g & me) != 0u && (__popc(g & lower) & 1) == 0;
        const bool take = even && above != 0u;
        const int src = take ? __ffs(above) - 1 : lane;
#pragma unroll
        for (int i = 0; i < 12; ++i) {
            const float o = __shfl_sync(full, v[i], src);
            if (take) v[i] += o;
        }
        g &= __ballot_sync(full, even);
    }
    return key >= 0 && (grp & lower) == 0u;
}

__global__ void __launch_bounds__(kLutThreads, 1)
    lut_grad_kernel(BwdArgs a, float *__restrict__ lut_part, float *__restrict__ sums_part)
{
    pdl_enter();
    extern __shared__ __align__(16) float sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = warp / 3, pair = warp - grp * 3;
    const int A = pair == 2 ? 1 : 0, Bx = pair == 0 ? 1 : 2;  // axes of the pair
    const int D = a.D, DD = D * D, tf = lut_table_floats(D);
    float *tab = sm + warp * tf;  // [D][D][3] of this warp's pair
    float4 *qv = reinterpret_cast<float4 *>(sm + kLutWarps * tf + warp * kLutQueueFloats);  // [3][kLutQueue]
    int *qk = reinterpret_cast<int *>(qv + 3 * kLutQueue);                                   // [kLutQueue]
    float *sums = sm + kLutWarps * (tf + kLutQueueFloats);                                   // [kLutGroups][4]
    const size_t plane = static_cast<size_t>(a.H) * a.W;
    const float fD1 = static_cast<float>(D - 1), fD2 = static_cast<float>(D - 2);
    const int strips = (a.W + kLutTileW - 1) / kLutTileW;
    const long long per_image = static_cast<long long>(strips) * a.H;
    const long long c1 = lut_share(per_image * a.B, gridDim.x, blockIdx.x + 1);
    for (long long c0 = lut_share(per_image * a.B, gridDim.x, blockIdx.x); c0 < c1;) {
        // this image's part of the share: units [u0, u1) of image b
        const int b = static_cast<int>(c0 / per_image);
        const long long u0 = c0 - b * per_image, u1 = min(c1 - b * per_image, per_image);
        c0 = b * per_image + u1;
        for (int e = threadIdx.x; e < kLutWarps * tf / 4; e += kLutThreads)
            reinterpret_cast<float4 *>(sm)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();

        const float *xa = a.x + (static_cast<size_t>(b) * 3 + A) * plane, *xbp = a.x + (static_cast<size_t>(b) * 3 + Bx) * plane;
        const float *gb = a.dy + static_cast<size_t>(b) * 3 * plane;
        const long long t0 = u0 + (u1 - u0) * grp / kLutGroups, t1 = u0 + (u1 - u0) * (grp + 1) / kLutGroups;
        const int my_rows = static_cast<int>(t1 - t0);

        float acc[2][12];  // [column][corner * 3 + channel]
        int acc_key[2] = {-1, -1};
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int i = 0; i < 12; ++i) acc[k][i] = 0.f;
        int qn = 0;  // queued sums
        float dysum[3] = {0.f, 0.f, 0.f};

        // adds the sums of the lanes with key >= 0 to the table
        auto add_batch = [&](int key, float (&v)[12]) {
            const bool leader = merge_equal_keys(key, v);
            const int off[4] = {0, 3 * D, 3, 3 * D + 3};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (leader) {
                    float *t = tab + key * 3 + off[q];
                    const float u0 = t[0], u1 = t[1], u2 = t[2];
                    t[0] = u0 + v[q * 3];
                    t[1] = u1 + v[q * 3 + 1];
                    t[2] = u2 + v[q * 3 + 2];
                }
                __syncwarp();
            }
        };
        auto drain = [&]() {
            float w[12];
            int k = -1;
            __syncwarp();
            if (lane < qn) {
                const float4 q0 = qv[lane], q1 = qv[kLutQueue + lane], q2 = qv[2 * kLutQueue + lane];
                w[0] = q0.x;
                w[1] = q0.y;
                w[2] = q0.z;
                w[3] = q0.w;
                w[4] = q1.x;
                w[5] = q1.y;
                w[6] = q1.z;
                w[7] = q1.w;
                w[8] = q2.x;
                w[9] = q2.y;
                w[10] = q2.z;
                w[11] = q2.w;
                k = qk[lane];
            } else {
#pragma unroll
                for (int i = 0; i < 12; ++i) w[i] = 0.f;
            }
            qn = 0;
            add_batch(k, w);
        };
        // the sums v of the lanes with key >= 0 are finished
        auto finish = [&](int key, float (&v)[12]) {
            const unsigned int done = __ballot_sync(0xffffffffu, key >= 0);
            const int cnt = __popc(done);
            if (cnt >= kLutDirect) {
                add_batch(key, v);
                return;
            }
            if (qn + cnt > kLutQueue) drain();
            if (key >= 0) {
                const int s = qn + __popc(done & ((1u << lane) - 1u));
                qv[s] = make_float4(v[0], v[1], v[2], v[3]);
                qv[kLutQueue + s] = make_float4(v[4], v[5], v[6], v[7]);
                qv[2 * kLutQueue + s] = make_float4(v[8], v[9], v[10], v[11]);
                qk[s] = key;
            }
            qn += cnt;
        };

        struct Row {
            float pa[2], pb[2], g[3][2];
            int n;  // this lane's columns: 0, 1 or 2
        };
        // rows are loaded one ahead of their use, from the cursor (strip, row)
        int ls = static_cast<int>(t0 / a.H), lr = static_cast<int>(t0 - ls * static_cast<long long>(a.H)), loaded = 0;
        auto load = [&](Row &o) {
            const int x = ls * kLutTileW + lane;
            o.n = loaded < my_rows ? (x < a.W) + (x + 32 < a.W) : 0;
            const size_t off = static_cast<size_t>(lr) * a.W + x;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const bool in = k < o.n;
                o.pa[k] = in ? __ldcs(xa + off + 32 * k) : 0.f;
                o.pb[k] = in ? __ldcs(xbp + off + 32 * k) : 0.f;
#pragma unroll
                for (int c = 0; c < 3; ++c) o.g[c][k] = in ? __ldcs(gb + c * plane + off + 32 * k) : 0.f;
            }
            ++loaded;
            if (++lr == a.H) {
                lr = 0;
                ++ls;
            }
        };
        Row cur, nxt;
        load(cur);
        for (int r = 0; r < my_rows; ++r) {
            load(nxt);
            float da[2], db[2];
            int key[2];
            bool change[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int ia = cell_of(__saturatef(cur.pa[k]), fD1, fD2, da[k]);
                const int ib = cell_of(__saturatef(cur.pb[k]), fD1, fD2, db[k]);
                key[k] = ia * D + ib;
                change[k] = k < cur.n && key[k] != acc_key[k];
            }
            if (__any_sync(0xffffffffu, change[0] || change[1])) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    finish(change[k] ? acc_key[k] : -1, acc[k]);
                    if (change[k]) {
#pragma unroll
                        for (int i = 0; i < 12; ++i) acc[k][i] = 0.f;
                        acc_key[k] = key[k];
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float w[4] = {(1.f - da[k]) * (1.f - db[k]), da[k] * (1.f - db[k]), (1.f - da[k]) * db[k], da[k] * db[k]};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    dysum[c] += cur.g[c][k];
                    // a column outside the image adds nothing (its dy is 0)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[k][q * 3 + c] = fmaf(cur.g[c][k], w[q], acc[k][q * 3 + c]);
                }
            }
            cur = nxt;
        }
        finish(acc_key[0], acc[0]);
        finish(acc_key[1], acc[1]);
        drain();

        // sum of dy_c: the pair-0 warps' totals (every pair warp of a group sees the same pixels)
#pragma unroll
        for (int c = 0; c < 3; ++c) dysum[c] = warp_sum(dysum[c]);
        if (lane == 0 && pair == 0) {
#pragma unroll
            for (int c = 0; c < 3; ++c) sums[grp * 4 + c] = dysum[c];
        }
        __syncthreads();
        // CTA partial [c][pair][vertex]: sum the groups in order
        const size_t slot = lut_slot(static_cast<int>(blockIdx.x), b, a.seg);
        float *out = lut_part + slot * 9 * DD;
        for (int e = threadIdx.x; e < 9 * DD; e += kLutThreads) {
            const int c = e / (3 * DD), r = e - c * 3 * DD, q = r / DD, vtx = r - q * DD;
            float s = 0.f;
#pragma unroll
            for (int g = 0; g < kLutGroups; ++g) s += sm[(g * 3 + q) * tf + vtx * 3 + c];
            out[e] = s;
        }
        if (threadIdx.x < 3) {
            float s = 0.f;
            for (int g = 0; g < kLutGroups; ++g) s += sums[g * 4 + threadIdx.x];
            sums_part[slot * 3 + threadIdx.x] = s;
        }
        __syncthreads();  // the tables are cleared for the next image
    }
}

// ---------------------------------------------------------------------------
// Grid gradients per output channel c (folded planes F_c = sum_{k=c mod 3}
// w_k g_k): dFxy_c[iy][ix], dFxc_c[ix][j], dFyc_c[iy][j].
// Blocks: 128-px column strip x BH rows (host plan); warp (group g, channel c)
// owns a contiguous run of rows of one channel.  Output per block: xy
// [nvy][nvx][3], xc [3][nvx][Dsc], yc [3][nvy][Dsc] in block-local indexing.
//
// All three planes of a channel spread the same two numbers per pixel, v0 =
// dy (1 - e) at intensity vertex j and v1 = dy e at j + 1.  A lane owns four
// adjacent columns of the strip and walks down its warp's rows, so
//   xc: a column's x weights are fixed; its sums over the rows go to the
//       column's own bins X[j][column] and are spread over the x vertices once
//       per block;
//   yc: the rows of one y-cell share their two vertices; the lane adds
//       (v (1 - dy), v dy) to its own bins Y[j][lane], which are summed over
//       the lanes when the y-cell changes;
//   xy: sum dy_c (1 - dy) and sum dy_c dy stay in registers per column and
//       are spread over the x vertices when the y-cell changes.
// The bank of every bin is the lane's own, so the updates are conflict-free
// and need no match, tree or barrier; every sum has one owner and a fixed
// order (bitwise repeatable).  Two y moments (not one bin row per image row)
// keep the lane sums off the per-row path; four columns per lane share one Y.
// One channel per warp, because a warp's bins (13 KB at Dsc = 17) bound the
// warps of an SM: 15 warps, where warps of three channels left 5 and the
// kernel waited on its own latency (361 us on 8 x 1920x1080).
// Measured on 8 x 1920x1080, grids at 1/8 resolution: 204 us, the shared-memory
// pipe at 56 % and the issue slots at 50 %; 655 us when each pixel went through
// a warp scatter (match, rank tree, leader's update) per channel.
// ---------------------------------------------------------------------------
struct GridPlan {
    int BH, bands, nblk;   // per image
    int nvx, nvy, rpw, nvyw;  // maxima
    int blk_stride;        // floats per block partial
    int groups;            // row groups of a block (one warp per channel each)
};

__host__ __device__ inline int grid_block_floats(int nvx, int nvy, int Dsc)
{
    return 3 * nvy * nvx + 3 * nvx * Dsc + 3 * nvy * Dsc;
}

constexpr int kGridGroups = 5;
constexpr int kGridThreads = 3 * kGridGroups * 32;

// floats of one warp: Y (at least the 2 x 128 staging of the xy flush), X,
// then the warp's yc and xy vertex rows
__host__ __device__ inline int grid_y_floats(int Dsc) { return Dsc * 64 > 2 * kTileW ? Dsc * 64 : 2 * kTileW; }
__host__ __device__ inline int grid_warp_floats(int nvx, int nvyw, int Dsc)
{
    return grid_y_floats(Dsc) + Dsc * kTileW + ((nvyw * (Dsc + nvx) + 3) & ~3);
}
// floats shared by the block: column offsets, first column of each x-cell
__host__ __device__ inline int grid_shared_floats(int nvx) { return kTileW + ((nvx + 1 + 3) & ~3); }

// Sums of 128 per-column values (column col at (col & 3) * 32 + (col >> 2))
// over the x vertices of the block: vertex v takes the columns of cell v with
// weight 1 - d and those of cell v - 1 with weight d.  Lanes are (part,
// vertex) pairs: each adds a contiguous part of its vertex's columns in order,
// the parts are combined by a butterfly.  store(v, sum) is called by part 0.
template <class Store>
__device__ __forceinline__ void spread_columns(const float *row, const float *cold, const int *cs, int nvx,
                                               Store store)
{
    const int lane = threadIdx.x & 31;
    int nvp = 2;
    while (nvp < nvx && nvp < 32) nvp <<= 1;
    const int parts = 32 / nvp, part = lane / nvp;
    for (int v0 = 0; v0 < nvx; v0 += nvp) {
        const int v = v0 + (lane & (nvp - 1));
        float s = 0.f;
        if (v < nvx) {
            const int lo = cs[max(v - 1, 0)], mid = cs[v], hi = cs[min(v + 1, nvx)];
            const int len = (hi - lo + parts - 1) / parts;
            const int c0 = lo + part * len, c1 = min(c0 + len, hi);
            for (int col = c0; col < c1; ++col) {
                const float d = cold[col], w = col < mid ? d : 1.f - d;
                s = fmaf(row[(col & 3) * 32 + (col >> 2)], w, s);
            }
        }
        for (int o = nvp; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (part == 0 && v < nvx) store(v, s);
    }
}

__global__ void __launch_bounds__(kGridThreads, 1)
    grid_grad_kernel(BwdArgs a, GridPlan gp, float *__restrict__ grid_part)
{
    pdl_enter();
    extern __shared__ __align__(16) float sm[];
    __shared__ int wy_off[kGridGroups], wy_n[kGridGroups];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = gp.groups * 3, nthr = nw * 32;
    const int grp = warp / 3, c = warp - grp * 3;
    const int b = blockIdx.y, lb = blockIdx.x;
    const int band = lb / a.strips, strip = lb - band * a.strips;
    const int x0 = strip * kTileW, y0 = band * gp.BH;
    const int rows = min(gp.BH, a.H - y0);
    if (rows <= 0) return;
    const int Dsc = a.Dsc;
    // block footprint
    int ixlo, ixhi, iylo, iyhi;
    float t;
    spatial_cell(x0, a.W, a.Dsx, a.rW1, ixlo, t);
    spatial_cell(min(x0 + kTileW - 1, a.W - 1), a.W, a.Dsx, a.rW1, ixhi, t);
    spatial_cell(y0, a.H, a.Dsy, a.rH1, iylo, t);
    spatial_cell(y0 + rows - 1, a.H, a.Dsy, a.rH1, iyhi, t);
    const int nvx = min(min(ixhi + 1, a.Dsx - 1) - ixlo + 1, gp.nvx);
    const int nvy = min(min(iyhi + 1, a.Dsy - 1) - iylo + 1, gp.nvy);
    // this warp's rows and their footprint
    const int rpw = (rows + gp.groups - 1) / gp.groups;
    const int wr0 = min(grp * rpw, rows), wr1 = min(wr0 + rpw, rows);
    int wylo = iylo, wyhi = iylo;
    if (wr1 > wr0) {
        spatial_cell(y0 + wr0, a.H, a.Dsy, a.rH1, wylo, t);
        spatial_cell(y0 + wr1 - 1, a.H, a.Dsy, a.rH1, wyhi, t);
    }
    const int nvyw = min(min(wyhi + 1, a.Dsy - 1) - wylo + 1, gp.nvyw);

    float *cold = sm;                                // [kTileW]
    int *cs = reinterpret_cast<int *>(sm + kTileW);  // [nvx + 1]
    float *wbase = sm + grid_shared_floats(gp.nvx);
    const int wf = grid_warp_floats(gp.nvx, gp.nvyw, Dsc);
    const int yf = grid_y_floats(Dsc), xf = Dsc * kTileW;
    float *wt = wbase + warp * wf;
    float2 *Y = reinterpret_cast<float2 *>(wt);  // [Dsc][32 lanes]
    float *X = wt + yf;                          // [Dsc][4 x 32 columns]
    float *tyc = X + xf;                         // [nvyw][Dsc]
    float *txy = tyc + gp.nvyw * Dsc;            // [nvyw][nvx]
    for (int e = threadIdx.x; e < nw * wf / 4; e += nthr)
        reinterpret_cast<float4 *>(wbase)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    // column offsets and the first column of each x-cell (cells 0 .. nvx - 2)
    const int ncols = min(kTileW, a.W - x0);
    for (int col = threadIdx.x; col < ncols; col += nthr) {
        int ix, ixp = -1;
        float d, dp;
        spatial_cell(x0 + col, a.W, a.Dsx, a.rW1, ix, d);
        ix = max(0, min(ix - ixlo, nvx - 2));
        if (col > 0) {
            spatial_cell(x0 + col - 1, a.W, a.Dsx, a.rW1, ixp, dp);
            ixp = max(0, min(ixp - ixlo, nvx - 2));
        }
        cold[col] = d;
        for (int v = ixp + 1; v <= ix; ++v) cs[v] = col;
        if (col == ncols - 1)
            for (int v = ix + 1; v <= nvx; ++v) cs[v] = ncols;
    }

    const size_t plane = static_cast<size_t>(a.H) * a.W;
    const int x = x0 + lane * 4;
    const int n = min(4, a.W - x);
    const float *xb = a.x + (static_cast<size_t>(b) * 3 + c) * plane + x;
    const float *gb = a.dy + (static_cast<size_t>(b) * 3 + c) * plane + x;
    const bool vec = a.vec && n == 4;
    const float fS1 = static_cast<float>(Dsc - 1), fS2 = static_cast<float>(Dsc - 2);
    // The lane's columns, and whether every lane's lie in at most two x-cells:
    // then a column adds to vertices i0 + cell and i0 + cell + 1, cell 0 or 1.
    float cd[4];
    bool c1[4];
    int i0 = 0, i3 = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int ix;
        spatial_cell(min(x + k, a.W - 1), a.W, a.Dsx, a.rW1, ix, cd[k]);
        if (k == 0) i0 = ix;
        c1[k] = ix != i0;
        i3 = ix;
    }
    const bool two_cells = __all_sync(0xffffffffu, i3 - i0 <= 1);
    __syncthreads();

    float sy0[4], sy1[4];  // xy sums of this lane's columns in the current y-cell
#pragma unroll
    for (int k = 0; k < 4; ++k) sy0[k] = sy1[k] = 0.f;
    // end of a y-cell (warp row iyw): Y over the lanes into tyc, the xy sums
    // over the columns into txy, both cleared
    auto flush = [&](int iyw) {
        __syncwarp();
        // an entry's lane sum starts at pair e mod 16 of the lanes and wraps:
        // neighbouring entries read different banks at a time
        for (int e = lane; e < Dsc; e += 32) {
            const float4 *row = reinterpret_cast<const float4 *>(Y) + e * 16;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
            for (int l = 0; l < 16; ++l) {
                const float4 q = row[(l + e) & 15];
                s0 += q.x + q.z;
                s1 += q.y + q.w;
            }
            float *t0 = tyc + iyw * Dsc + e;
            t0[0] += s0;
            t0[Dsc] += s1;
        }
        __syncwarp();
        float *r0 = txy + iyw * gp.nvx, *r1 = r0 + gp.nvx;
        if (two_cells) {
            // the lane's sums at vertices i0, i0 + 1 and i0 + 2, then every
            // vertex adds those of the lanes that touch it, in order
            float2 s[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float w1 = cd[k], w0 = 1.f - w1;
                const float2 lo = make_float2(sy0[k] * w0, sy1[k] * w0), hi = make_float2(sy0[k] * w1, sy1[k] * w1);
                const int q = c1[k] ? 1 : 0;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    if (i == q) s[i] = make_float2(s[i].x + lo.x, s[i].y + lo.y);
                    if (i == q + 1) s[i] = make_float2(s[i].x + hi.x, s[i].y + hi.y);
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) Y[q * 32 + lane] = s[q];
            __syncwarp();
            for (int v = lane; v < nvx; v += 32) {
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int i = v - q;  // lanes whose first column lies in cell i
                    if (i < 0 || i > nvx - 2) continue;
                    for (int l = (cs[i] + 3) >> 2; l < (cs[i + 1] + 3) >> 2; ++l) {
                        const float2 u = Y[q * 32 + l];
                        s0 += u.x;
                        s1 += u.y;
                    }
                }
                r0[v] += s0;
                r1[v] += s1;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                wt[k * 32 + lane] = sy0[k];
                wt[kTileW + k * 32 + lane] = sy1[k];
            }
            __syncwarp();
            spread_columns(wt, cold, cs, nvx, [&](int v, float s) { r0[v] += s; });
            __syncwarp();
            spread_columns(wt + kTileW, cold, cs, nvx, [&](int v, float s) { r1[v] += s; });
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) sy0[k] = sy1[k] = 0.f;
        __syncwarp();
        for (int e = lane; e < yf / 4; e += 32) reinterpret_cast<float4 *>(wt)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
    };

    auto load = [&](int r, float4 &p, float4 &g) {
        p = g = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < wr1 && n > 0) {
            const size_t off = static_cast<size_t>(y0 + r) * a.W;
            p = PixIO<float>::load(xb + off, n, vec);
            g = PixIO<float>::load(gb + off, n, vec);
        }
    };
    int iy_acc = -1, cy = 0;
    float cdy = 0.f;
    auto row = [&](int r, const float4 &p, const float4 &g4) {
        // y-cells of the next 32 rows, one per lane
        const int ri = (r - wr0) & 31;
        if (ri == 0) {
            spatial_cell(min(y0 + r + lane, a.H - 1), a.H, a.Dsy, a.rH1, cy, cdy);
            cy = max(0, min(cy - wylo, nvyw - 2));
        }
        const int iyw = __shfl_sync(0xffffffffu, cy, ri);
        const float dy = __shfl_sync(0xffffffffu, cdy, ri), dy0 = 1.f - dy;
        if (iyw != iy_acc) {
            if (iy_acc >= 0) flush(iy_acc);
            iy_acc = iyw;
        }
        int j[4];
        float v0[4], v1[4], u0[4], u1[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float g = get(g4, k);
            float e;
            j[k] = cell_of(__saturatef(get(p, k)), fS1, fS2, e);
            v0[k] = g * (1.f - e);
            v1[k] = g * e;
            sy0[k] = fmaf(g, dy0, sy0[k]);
            sy1[k] = fmaf(g, dy, sy1[k]);
            const float *xp = X + j[k] * kTileW + k * 32 + lane;
            u0[k] = xp[0];
            u1[k] = xp[kTileW];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float *xp = X + j[k] * kTileW + k * 32 + lane;
            xp[0] = u0[k] + v0[k];
            xp[kTileW] = u1[k] + v1[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float2 *yp = Y + j[k] * 32 + lane;
            const float2 q0 = yp[0], q1 = yp[32];
            yp[0] = make_float2(fmaf(v0[k], dy0, q0.x), fmaf(v0[k], dy, q0.y));
            yp[32] = make_float2(fmaf(v1[k], dy0, q1.x), fmaf(v1[k], dy, q1.y));
        }
    };
    float4 pa, ga, pb, gb4;
    load(wr0, pa, ga);
    for (int r = wr0; r < wr1; r += 2) {
        load(r + 1, pb, gb4);
        row(r, pa, ga);
        load(r + 2, pa, ga);
        if (r + 1 < wr1) row(r + 1, pb, gb4);
    }
    if (iy_acc >= 0) flush(iy_acc);
    if (lane == 0 && c == 0) {
        wy_off[grp] = wylo - iylo;
        wy_n[grp] = wr1 > wr0 ? nvyw : 0;
    }
    __syncthreads();
    // block partial: the row groups in order
    float *out = grid_part + (static_cast<size_t>(b) * gp.nblk + lb) * gp.blk_stride;
    float *oxy = out, *oxc = out + 3 * gp.nvy * gp.nvx, *oyc = oxc + 3 * gp.nvx * Dsc;
    const float *wx = wbase + yf, *wyc = wx + xf, *wxy = wyc + gp.nvyw * Dsc;  // warp 0's tables
    for (int e = threadIdx.x; e < nvy * nvx * 3; e += nthr) {
        const int iyb = e / (nvx * 3), q = e - iyb * nvx * 3, v = q / 3, ch = q - v * 3;
        float s = 0.f;
        for (int g = 0; g < gp.groups; ++g) {
            const int iw = iyb - wy_off[g];
            if (iw >= 0 && iw < wy_n[g]) s += wxy[(g * 3 + ch) * wf + iw * gp.nvx + v];
        }
        oxy[iyb * gp.nvx * 3 + q] = s;
    }
    for (int e = threadIdx.x; e < 3 * nvy * Dsc; e += nthr) {
        const int ch = e / (nvy * Dsc), q = e - ch * nvy * Dsc, iyb = q / Dsc, j = q - iyb * Dsc;
        float s = 0.f;
        for (int g = 0; g < gp.groups; ++g) {
            const int iw = iyb - wy_off[g];
            if (iw >= 0 && iw < wy_n[g]) s += wyc[(g * 3 + ch) * wf + iw * Dsc + j];
        }
        oyc[(ch * gp.nvy + iyb) * Dsc + j] = s;
    }
    // X of all groups, summed into group 0's, then spread over the x vertices
    for (int e = threadIdx.x; e < 3 * (xf / 4); e += nthr) {
        const int ch = e / (xf / 4), i = e - ch * (xf / 4);
        float4 *x4 = reinterpret_cast<float4 *>(wbase + ch * wf + yf) + i;
        float4 s = *x4;
        for (int g = 1; g < gp.groups; ++g) {
            const float4 q = reinterpret_cast<const float4 *>(wx + (g * 3 + ch) * wf)[i];
            s.x += q.x;
            s.y += q.y;
            s.z += q.z;
            s.w += q.w;
        }
        *x4 = s;
    }
    __syncthreads();
    for (int q = warp; q < 3 * Dsc; q += nw) {
        const int ch = q >= Dsc ? (q >= 2 * Dsc ? 2 : 1) : 0, j = q - ch * Dsc;
        spread_columns(wx + ch * wf + j * kTileW, cold, cs, nvx,
                       [&](int v, float s) { oxc[(ch * gp.nvx + v) * Dsc + j] = s; });
    }
}

// ---------------------------------------------------------------------------
// LUT finalize: one CTA per (table c*3+pair, image).  The image's partials are
// summed in up to kFinParts contiguous parts, side by side, kFinBatch loads at a
// time, then the parts in order: two images' 152 partials on 18 CTAs were bound
// by the latency of one chain of loads per vertex (76 us at 2 x 342x628; 17 us at
// 8 x 1920x1080 and at 64 x 256x256 as it is, 27 and 20 before).  One thread
// works out the image's slots: with that in every thread the kernel took 45
// registers instead of 32, two CTAs of 512 threads per SM instead of four, and
// svdlut_backward at 64 x 256x256 340 us instead of 337.
// ---------------------------------------------------------------------------
constexpr int kFinMaxThreads = 1024, kFinParts = 8, kFinBatch = 8;

__device__ inline float block_sum(float v, float *red)
{
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float s = 0.f;
    for (int w = 0; w < static_cast<int>(blockDim.x) / 32; ++w) s += red[w];
    return s;
}

struct FinArgs {
    const float *U, *S, *V, *lw;
    float *dU, *dS, *dV, *dlw;
    int D, R, B, G, seg;  // G: CTAs of the LUT pass; seg: lut_segment
    long long per_image;  // its work units per image
};

__host__ __device__ inline int fin_smem_floats(int D, int R) { return kFinParts * D * D + 3 * D * R + R + kFinMaxThreads / 32; }

__global__ void __launch_bounds__(kFinMaxThreads)
    lut_finalize_kernel(FinArgs f, const float *__restrict__ lut_part, const float *__restrict__ sums_part)
{
    pdl_enter();
    extern __shared__ __align__(16) float sm[];
    const int nthr = blockDim.x;
    const int cp = blockIdx.x, b = blockIdx.y, c = cp / 3, pair = cp - c * 3;
    const int D = f.D, R = f.R, DD = D * D, DR = D * R;
    __shared__ int slots[2];  // the image's
    if (threadIdx.x == 0) lut_slots(f.per_image, f.B, f.G, f.seg, b, slots[0], slots[1]);
    __syncthreads();
    const int s0 = slots[0], s1 = slots[1];
    float *G = sm;  // [kFinParts][DD]: the parts' sums, then G = the gradient of the table in part 0
    float *U = sm + kFinParts * DD, *V = U + DR, *Q = V + DR, *S = Q + DR, *red = S + R;  // Q[i][r] = sum_j dT[i][j] V[j][r]
    const size_t t = static_cast<size_t>(b) * 9 + cp;
    for (int e = threadIdx.x; e < DR; e += nthr) {
        U[e] = f.U[t * DR + e];
        V[e] = f.V[t * DR + e];
    }
    if (threadIdx.x < R) S[threadIdx.x] = f.S[t * R + threadIdx.x];
    const float w = f.lw[static_cast<size_t>(b) * 12 + c * 4 + pair];
    const int n = s1 - s0, parts = max(1, min(kFinParts, n / kFinBatch));
    for (int it = threadIdx.x; it < parts * DD; it += nthr) {
        const int part = it / DD, e = it - part * DD;
        const int q1 = s0 + n * (part + 1) / parts;
        const float *src = lut_part + cp * DD + e;
        float s = 0.f;
        for (int q = s0 + n * part / parts; q < q1; q += kFinBatch) {
            float v[kFinBatch];
#pragma unroll
            for (int u = 0; u < kFinBatch; ++u) v[u] = q + u < q1 ? src[static_cast<size_t>(q + u) * 9 * DD] : 0.f;
#pragma unroll
            for (int u = 0; u < kFinBatch; ++u) s += v[u];
        }
        G[it] = s;
    }
    __syncthreads();
    // G, and dw = <G, T>
    float part = 0.f;
    for (int e = threadIdx.x; e < DD; e += nthr) {
        float g = G[e];
        for (int p = 1; p < parts; ++p) g += G[p * DD + e];
        G[e] = g;
        const int i = e / D, j = e - i * D;
        float tv = 0.f;
        for (int r = 0; r < R; ++r) tv = fmaf(U[i * R + r] * S[r], V[j * R + r], tv);
        part = fmaf(g, tv, part);
    }
    const float dw = block_sum(part, red);
    if (threadIdx.x == 0 && f.dlw) {
        f.dlw[static_cast<size_t>(b) * 12 + c * 4 + pair] = dw;
        if (pair == 0) {
            float s = 0.f;
#pragma unroll 8
            for (int q = s0; q < s1; ++q) s += sums_part[static_cast<size_t>(q) * 3 + c];
            f.dlw[static_cast<size_t>(b) * 12 + c * 4 + 3] = s;
        }
    }
    // Q = (w G) V; dU = Q diag(S); dV = (w G)^T U diag(S): items 0 .. DR - 1 and DR .. 2 DR - 1
    for (int it = threadIdx.x; it < 2 * DR; it += nthr) {
        const bool vside = it >= DR;
        const int e = vside ? it - DR : it, i = e / R, r = e - i * R;
        const float *g = G + (vside ? i : i * D), *m = (vside ? U : V) + r;
        const int gs = vside ? D : 1;
        float s = 0.f;
#pragma unroll 8
        for (int j = 0; j < D; ++j) s = fmaf(g[j * gs], m[j * R], s);
        if (!vside) Q[e] = w * s;
        float *out = vside ? f.dV : f.dU;
        if (out) out[t * DR + e] = w * s * S[r];
    }
    __syncthreads();
    // dS_r = sum_i U[i][r] Q[i][r]
    if (f.dS && threadIdx.x < R) {
        const int r = threadIdx.x;
        float s = 0.f;
        for (int i = 0; i < D; ++i) s = fmaf(U[i * R + r], Q[i * R + r], s);
        f.dS[t * R + r] = s;
    }
}

// ---------------------------------------------------------------------------
// grid reduce and finalize, fused.  A CTA takes a slice of kGRChunk vertices
// of the folded planes xy, xc or yc of one image, a thread one vertex of all
// three output channels (their blocks and offsets are the same).  It sums the
// partials of the blocks whose footprint holds the vertex (bands, then strips,
// in order), which is dF_c at that vertex; then for every grid k, c = k mod 3,
// it writes dg^k_plane = w^k_plane dF_c (Supp. Eqs. 21-22: grid k feeds channel
// k mod 3 with weight w^k_plane), and the sum of dF_c g^k_plane over the slice
// is a partial of dgrid_w[k][plane].  grid_wsum_kernel sums those over the
// slices in order.  Bound by latency and by finding the blocks (divisions):
// the partials of kGRBatch blocks are loaded, then added; one channel per
// thread and one load after another took 41 us at 2 x 342x628 (22 bands) and
// 47 at 8 x 1920x1080, 29 as it is.
// ---------------------------------------------------------------------------
constexpr int kGRThreads = 512, kGRChunk = kGRThreads;
constexpr int kGRBatch = 4;  // blocks in flight per vertex

struct GridRed {
    int B, H, W, K, Dsx, Dsy, Dsc, strips;
    float rW1, rH1;
    GridPlan gp;
    int sl[3];  // slices per plane: xy, xc, yc
    int smax;   // max(sl)
    const float *gxy, *gxc, *gyc, *gw;
    float *dgxy, *dgxc, *dgyc;  // any may be null
    float *wpart;               // [B][3 planes][K][smax] partial sums of dgrid_w, or null
};

// block footprint along one axis: first vertex and count (as grid_grad_kernel)
__device__ __forceinline__ void axis_span(int p0, int cnt, int n, int Ds, float rn1, int vmax, int &lo, int &nv)
{
    int hi;
    float t;
    spatial_cell(p0, n, Ds, rn1, lo, t);
    spatial_cell(p0 + cnt - 1, n, Ds, rn1, hi, t);
    nv = min(min(hi + 1, Ds - 1) - lo + 1, vmax);
}

// range of strips / bands whose footprint may contain vertex v (pixel range
// between the neighbouring vertices)
__device__ __forceinline__ void cover_range(int v, int n, int Ds, int unit, int nunits, int &u0, int &u1)
{
    if (n <= 1) {
        u0 = 0;
        u1 = nunits - 1;
        return;
    }
    // a / d for 0 <= a, 1 <= d: a 32-bit division whenever a fits
    auto div = [](long long a, int d) -> long long {
        return a <= 0xffffffffLL ? static_cast<long long>(static_cast<unsigned int>(a) / static_cast<unsigned int>(d))
                                 : a / d;
    };
    const long long lo = div(static_cast<long long>(max(v - 1, 0)) * (n - 1), Ds - 1);
    const long long hi = div(static_cast<long long>(min(v + 1, Ds - 1)) * (n - 1) + (Ds - 2), Ds - 1);
    u0 = max(0, static_cast<int>(div(lo, unit)) - 1);
    u1 = min(nunits - 1, static_cast<int>(div(hi, unit)) + 1);
}

__host__ __device__ inline int grid_plane_size(int plane, int Dsx, int Dsy, int Dsc)
{
    return plane == 0 ? Dsy * Dsx : (plane == 1 ? Dsx * Dsc : Dsy * Dsc);
}

__global__ void __launch_bounds__(kGRThreads, 3)
    grid_reduce_kernel(GridRed g, const float *__restrict__ grid_part)
{
    pdl_enter();
    extern __shared__ int gtab[];  // ylo[bands], nvy[bands], xlo[strips], nvx[strips]; then the warps' sums [][K]
    const GridPlan &gp = g.gp;
    const int b = blockIdx.y;
    int slice = blockIdx.x, plane = 0;  // blockIdx.x -> (plane, slice)
    while (plane < 2 && slice >= g.sl[plane]) slice -= g.sl[plane++];
    int *ylo = gtab, *nvy = gtab + gp.bands, *xlo = nvy + gp.bands, *nvx = xlo + g.strips;
    for (int t = threadIdx.x; t < gp.bands + g.strips; t += kGRThreads) {
        if (t < gp.bands) {
            const int y0 = t * gp.BH, rows = min(gp.BH, g.H - y0);
            if (rows > 0) axis_span(y0, rows, g.H, g.Dsy, g.rH1, gp.nvy, ylo[t], nvy[t]);
            else ylo[t] = nvy[t] = 0;
        } else {
            const int st = t - gp.bands, x0 = st * kTileW;
            axis_span(x0, min(kTileW, g.W - x0), g.W, g.Dsx, g.rW1, gp.nvx, xlo[st], nvx[st]);
        }
    }
    __syncthreads();
    const int Dsx = g.Dsx, Dsy = g.Dsy, Dsc = g.Dsc, K = g.K;
    const int n = grid_plane_size(plane, Dsx, Dsy, Dsc), ncol = plane == 0 ? Dsx : Dsc;
    const float *gsrc = plane == 0 ? g.gxy : (plane == 1 ? g.gxc : g.gyc);
    float *gdst = plane == 0 ? g.dgxy : (plane == 1 ? g.dgxc : g.dgyc);
    const int e = slice * kGRChunk + threadIdx.x;
    const bool in = e < n;
    float s[3] = {0.f, 0.f, 0.f};
    if (in) {
        // xy: (iy, ix); xc: (ix, j); yc: (iy, j)
        const int r = e / ncol, col = e - r * ncol;
        const int iy = plane == 1 ? -1 : r, ix = plane == 0 ? col : (plane == 1 ? r : -1);
        int s0 = 0, s1 = g.strips - 1, b0 = 0, b1 = gp.bands - 1;
        if (ix >= 0) cover_range(ix, g.W, Dsx, kTileW, g.strips, s0, s1);
        if (iy >= 0) cover_range(iy, g.H, Dsy, gp.BH, gp.bands, b0, b1);
        // offset in a block partial of the block's first vertex, strides of the
        // vertex and of the channel
        const int oxc = 3 * gp.nvy * gp.nvx, oyc = oxc + 3 * gp.nvx * Dsc;
        const int base = plane == 0 ? 0 : (plane == 1 ? oxc + col : oyc + col);
        const int vy = plane == 0 ? 3 * gp.nvx : (plane == 1 ? 0 : Dsc), vx = plane == 0 ? 3 : (plane == 1 ? Dsc : 0);
        const int vc = plane == 0 ? 1 : (plane == 1 ? gp.nvx * Dsc : gp.nvy * Dsc);
        const int nb = (b1 - b0 + 1) * (s1 - s0 + 1);
        const float *img = grid_part + static_cast<size_t>(b) * gp.nblk * gp.blk_stride + base;
        int bd = b0, st = s0;
        for (int t = 0; t < nb; t += kGRBatch) {
            float v[kGRBatch][3];
#pragma unroll
            for (int u = 0; u < kGRBatch; ++u) {
                v[u][0] = v[u][1] = v[u][2] = 0.f;
                if (t + u < nb) {
                    const int dy = iy - ylo[bd], dx = ix - xlo[st], ny = nvy[bd];
                    if (ny > 0 && (iy < 0 || (dy >= 0 && dy < ny)) && (ix < 0 || (dx >= 0 && dx < nvx[st]))) {
                        const float *bp = img + static_cast<size_t>(bd * g.strips + st) * gp.blk_stride + dy * vy + dx * vx;
#pragma unroll
                        for (int c = 0; c < 3; ++c) v[u][c] = bp[c * vc];
                    }
                    if (++st > s1) {
                        st = s0;
                        ++bd;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kGRBatch; ++u)
#pragma unroll
                for (int c = 0; c < 3; ++c) s[c] += v[u][c];
        }
    }
    // the grids, three at a time (channels 0, 1, 2)
    float *red = reinterpret_cast<float *>(gtab);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int k0 = 0; k0 < K; k0 += 3) {
        float gv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int k = k0 + c;
            gv[c] = 0.f;
            if (k < K && in) {
                const size_t bk = static_cast<size_t>(b) * K + k;
                if (gdst) gdst[bk * n + e] = __ldg(g.gw + bk * 4 + plane) * s[c];
                if (g.wpart) gv[c] = __ldg(gsrc + bk * n + e) * s[c];
            }
        }
        if (!g.wpart) continue;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float t = warp_sum(gv[c]);
            if (lane == 0 && k0 + c < K) red[warp * K + k0 + c] = t;
        }
    }
    if (!g.wpart) return;
    __syncthreads();
    // the slice's partials of dgrid_w: the warps in order
    if (static_cast<int>(threadIdx.x) < K) {
        const int k = threadIdx.x;
        float t = 0.f;
        for (int w = 0; w < kGRThreads / 32; ++w) t += red[w * K + k];
        g.wpart[((static_cast<size_t>(b) * 3 + plane) * K + k) * g.smax + slice] = t;
    }
}

// dgrid_w[b][k] = (the slice partials of each plane summed in order, the sum
// of dy_{k mod 3} over the image from the LUT pass partials: the bias).
struct GridWsum {
    int B, K, G, seg, smax;
    int sl[3];
    float *dgw;
    long long per_image;
};

__global__ void grid_wsum_kernel(GridWsum f, const float *__restrict__ wpart, const float *__restrict__ sums_part)
{
    pdl_enter();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;  // (b, k, entry)
    if (t >= f.B * f.K * 4) return;
    const int q = t & 3, bk = t >> 2, b = bk / f.K, k = bk - b * f.K;
    float s = 0.f;
    if (q < 3) {
        const float *p = wpart + ((static_cast<size_t>(b) * 3 + q) * f.K + k) * f.smax;
#pragma unroll 8
        for (int i = 0; i < f.sl[q]; ++i) s += p[i];
    } else {
        int s0, s1;
        lut_slots(f.per_image, f.B, f.G, f.seg, b, s0, s1);
#pragma unroll 8
        for (int i = s0; i < s1; ++i) s += sums_part[static_cast<size_t>(i) * 3 + k % 3];
    }
    f.dgw[static_cast<size_t>(bk) * 4 + q] = s;
}

// ---------------------------------------------------------------------------
// host planning and workspace
// ---------------------------------------------------------------------------
struct BwdPlan {
    int G;             // LUT-pass CTAs
    long long units;   // its work units per image
    size_t lut_smem;   // bytes
    GridPlan gp;
    size_t grid_smem;  // bytes
    // workspace layout (bytes); the last part holds the per-image tables of
    // the dx pass (prep_kernel)
    size_t off_lut, off_sums, off_grid, off_wpart, off_prep, prep_img, total;
    int sl[3], smax;  // grid_reduce_kernel slices per channel plane (xy, xc, yc)
};

static size_t align256(size_t v) { return (v + 255) & ~static_cast<size_t>(255); }

// Opts kernel f into the largest dynamic shared memory its static shared
// memory leaves, once per device (calls from several threads are serialised).
static svdlut_status allow_dynamic_smem(const void *f, int max_optin, int device)
{
    static std::mutex mu;
    static std::vector<std::pair<int, const void *>> done;
    std::lock_guard<std::mutex> g(mu);
    for (const auto &e : done)
        if (e.first == device && e.second == f) return SVDLUT_OK;
    cudaFuncAttributes fa;
    SVDLUT_CUDA_TRY(cudaFuncGetAttributes(&fa, f));
    SVDLUT_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         max_optin - static_cast<int>(fa.sharedSizeBytes)));
    done.emplace_back(device, f);
    return SVDLUT_OK;
}

// Grid densities that the adjoint takes, a rule of the entry point and not what
// the kernel could hold: 16 warps' xy, xc and yc vertices of a block of BH rows,
// three channels each, in the shared memory (about one vertex per two pixels at
// Dsc = 17).  Whatever it takes fits as a block of one row (plan_grid): one row
// group's warps want 3 * (192 Dsc + nvyw (Dsc + nvx)) floats, and the rule bounds
// 48 * nvyw (Dsc + nvx) by the shared memory.
static bool grid_density_ok(int BH, int nvx, int H, int Dsy, int Dsc, size_t smem_limit)
{
    const int nvyw = span_bound((BH + kWarps - 1) / kWarps, H, Dsy);
    const size_t warp = (3 * (static_cast<size_t>(nvyw) * nvx + static_cast<size_t>(nvx + nvyw) * Dsc) + 3) & ~size_t(3);
    return sizeof(float) * kWarps * warp + 256 <= smem_limit;
}

// Workspace layout of a plan whose G and gp are set.
static void layout_backward(const svdlut_dims *d, int B, BwdPlan *pl)
{
    const int D = d->D_t;
    size_t off = 0;
    pl->off_lut = off;
    const size_t slots = lut_slot_count(pl->G, B);
    off = align256(off + sizeof(float) * slots * 9 * D * D);
    pl->off_sums = off;
    off = align256(off + sizeof(float) * slots * 3);
    pl->off_grid = off;
    off = align256(off + sizeof(float) * static_cast<size_t>(B) * pl->gp.nblk * pl->gp.blk_stride);
    pl->smax = 1;
    for (int q = 0; q < 3; ++q) {
        pl->sl[q] = (grid_plane_size(q, d->Dsx, d->Dsy, d->Dsc) + kGRChunk - 1) / kGRChunk;
        pl->smax = std::max(pl->smax, pl->sl[q]);
    }
    pl->off_wpart = off;
    off = align256(off + sizeof(float) * static_cast<size_t>(B) * 3 * std::max(d->K, 0) * pl->smax);
    pl->off_prep = off;
    pl->prep_img = prep_image_bytes(d);
    off += static_cast<size_t>(B) * pl->prep_img;
    pl->total = off;
}

// LUT pass: CTAs, at most max_g (one per SM) and with at most max_slots parts;
// estimated time = rows a group walks (its share of the batch's strips x rows,
// + a fixed cost of about 16 rows per CTA: clearing the tables, writing the
// partial) + a row's time per 24 partials of an image that lut_finalize_kernel
// sums.
static int plan_lut_ctas(int B, long long units, int max_g, size_t max_slots)
{
    const long long U = units * B;
    long long best_cost = -1;
    int best = 1;
    for (int G = 1; G <= std::min<long long>(U, max_g); ++G) {
        if (lut_slot_count(G, B) > max_slots) continue;
        const long long cost = 24 * (((U + G - 1) / G + kLutGroups - 1) / kLutGroups + 16) + (G + B - 1) / B;
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = G;
        }
    }
    return best;
}

// Grid pass of a plan whose G is set: blocks of 128 x BH with as many row
// groups as fit; bands minimise waves x (rows a warp walks + a fixed cost of
// about 8 rows per block: clearing the tables, summing the warps, writing the
// partial), ties go to the better-filled waves, and plans within ws_limit bytes
// go before larger ones.  smallest: the smallest workspace instead.  Blocks have
// at least about 16 rows; where the y vertices are so dense that no such block's
// row groups hold theirs (Dsc = 64: six per image row), the tallest block that
// fits.  False for densities that the adjoint does not take.
static bool plan_grid(const svdlut_dims *d, int B, int H, int W, int sm_count, size_t smem_limit, size_t ws_limit,
                      bool smallest, BwdPlan *pl)
{
    const int Dsc = d->Dsc;
    const int strips = (W + kTileW - 1) / kTileW, nvx = span_bound(kTileW, W, d->Dsx);
    const int max_bands = std::max(1, (H + kMinBlockH - 1) / kMinBlockH);
    BwdPlan best{};
    bool taken = false, fits = false;
    double best_score = -1e30;
    auto consider = [&](int BH) {
        BwdPlan q = *pl;
        GridPlan &gp = q.gp;
        gp.BH = BH;
        gp.bands = (H + BH - 1) / BH;
        gp.nvx = nvx;
        gp.nvy = span_bound(BH, H, d->Dsy);
        for (gp.groups = kGridGroups; gp.groups > 0; --gp.groups) {
            gp.rpw = (BH + gp.groups - 1) / gp.groups;
            gp.nvyw = span_bound(gp.rpw, H, d->Dsy);
            q.grid_smem = sizeof(float) * (static_cast<size_t>(grid_shared_floats(nvx)) +
                                           static_cast<size_t>(3 * gp.groups) * grid_warp_floats(nvx, gp.nvyw, Dsc));
            if (q.grid_smem + 256 <= smem_limit) break;  // + the kernel's static row offsets
        }
        if (gp.groups == 0) return;
        gp.nblk = strips * gp.bands;
        gp.blk_stride = grid_block_floats(nvx, gp.nvy, Dsc);
        layout_backward(d, B, &q);
        const long long T = static_cast<long long>(B) * strips * gp.bands;
        const double waves = std::ceil(static_cast<double>(T) / sm_count - 1e-9);
        const double fill = static_cast<double>(T) / (waves * sm_count);
        const double score = smallest ? -static_cast<double>(q.total)
                                      : -waves * (gp.rpw + 8) + 1e-3 * fill - (q.total > ws_limit ? 1e12 : 0.0);
        if (!fits || score > best_score + 1e-12) {
            best_score = score;
            best = q;
            fits = true;
        }
    };
    for (int bands = 1; bands <= max_bands; ++bands) {
        const int BH = (H + bands - 1) / bands;
        if (!grid_density_ok(BH, nvx, H, d->Dsy, Dsc, smem_limit)) continue;
        taken = true;
        consider(BH);
        if (fits && bands >= 4 * sm_count) break;
    }
    if (taken)
        for (int BH = std::min(H, kMinBlockH); BH > 0 && !fits; --BH) consider(BH);
    if (fits) *pl = best;
    return fits;
}

// ws_limit: bytes that the caller can give (svdlut_backward_noalloc's scratch;
// SIZE_MAX for svdlut_backward, whose caller allocates what the plan wants).  A
// plan beyond it gives way to one within it, if there is any: beside the smallest
// grid plan the LUT CTAs whose parts there is room for, then the best grid plan
// beside those.  CTAs that hold whole images, or images that are whole CTAs, want
// the fewest parts: 154 images of 256 x 256 leave room for 154 parts, 77 CTAs of
// two images each.
static svdlut_status plan_backward(const svdlut_dims *d, int B, int H, int W, int sm_count, size_t smem_limit,
                                   size_t ws_limit, BwdPlan *pl)
{
    pl->lut_smem = lut_grad_smem(d->D_t);
    if (pl->lut_smem > smem_limit) return fail(SVDLUT_ERR_UNSUPPORTED, "D_t=%d too large for the adjoint", d->D_t);
    pl->units = static_cast<long long>((W + kLutTileW - 1) / kLutTileW) * H;
    pl->G = plan_lut_ctas(B, pl->units, sm_count, SIZE_MAX);
    if (!plan_grid(d, B, H, W, sm_count, smem_limit, ws_limit, false, pl))
        return fail(SVDLUT_ERR_UNSUPPORTED, "grid vertices too dense for the adjoint's blocks");
    if (pl->total > ws_limit) {
        BwdPlan q = *pl;
        q.G = 1;
        plan_grid(d, B, H, W, sm_count, smem_limit, ws_limit, true, &q);
        if (q.total <= ws_limit) {
            const size_t per = sizeof(float) * (9 * static_cast<size_t>(d->D_t) * d->D_t + 3);
            size_t slots = static_cast<size_t>(B) + (ws_limit - q.total) / per;
            do {
                q.G = plan_lut_ctas(B, q.units, sm_count, slots--);
                layout_backward(d, B, &q);
            } while (q.total > ws_limit);  // the parts' alignment
            plan_grid(d, B, H, W, sm_count, smem_limit, ws_limit, false, &q);
            *pl = q;
        }
    }
    return SVDLUT_OK;
}

// The dx pass, N images per launch; with `tables` (B times prep_img bytes) the
// per-image tables are precomputed once (prep_kernel) instead of in every CTA:
// the instance that builds them spills registers, and loses 1 to 5 % at most
// sizes (77 -> 74 us for svdlut_backward at 2 x 224x106, 490 -> 477 at 11 x
// 514x1392; 337 -> 341 at 64 x 256x256).  One launch for 64 images of 256 x 256 instead of four of 16: the
// blocks of a launch fill the SMs once, and three tails and table launches go.
template <int N>
static svdlut_status dx_chunks(const svdlut_dims *dims, const svdlut_params *params, int B, int H, int W,
                               const float *x, const float *dy, float *dx, char *tables, size_t prep_img,
                               const DeviceInfo &di, cudaStream_t s)
{
    svdlut_status st = SVDLUT_OK;
    for (int b0 = 0; b0 < B; b0 += N) {
        LaunchArgs<N> a{};
        a.n = std::min(N, B - b0);
        for (int i = 0; i < a.n; ++i) {
            a.img[i] = make_desc(dims, params, b0 + i, H, W, SVDLUT_F32, x, dx);
            a.img[i].dy = dy + static_cast<size_t>(b0 + i) * 3 * H * W;
            a.img[i].vec = a.img[i].vec && aligned(a.img[i].dy, 16);
            if (tables) set_prep_tables(a.img[i], dims, tables + static_cast<size_t>(b0 + i) * prep_img);
        }
        size_t smem = 0;
        if ((st = plan_uniform(a, di.sm_count, static_cast<size_t>(di.max_smem_optin), &smem)) != SVDLUT_OK) return st;
        if (tables) {
            if ((st = launch_prep(a, di.sm_count, s)) != SVDLUT_OK) return st;
            a.pre = kPreAll;
        }
        if ((st = launch_apply(a, smem, SVDLUT_F32, s, 0, true)) != SVDLUT_OK) return st;
    }
    return SVDLUT_OK;
}

static svdlut_status check_backward_args(const svdlut_dims *dims, const svdlut_params *params, int B, int H,
                                         int W, const float *x, const float *dy)
{
    svdlut_status st = check_dims(dims);
    if (st != SVDLUT_OK) return st;
    if ((st = check_params(dims, params)) != SVDLUT_OK) return st;
    if (B < 1 || H < 1 || W < 1) return fail(SVDLUT_ERR_INVALID_ARG, "B=%d H=%d W=%d must be >= 1", B, H, W);
    if (!x || !dy) return fail(SVDLUT_ERR_INVALID_ARG, "x and dy are required");
    if (!aligned(x, 4) || !aligned(dy, 4)) return fail(SVDLUT_ERR_INVALID_ARG, "x and dy must be 4-byte aligned");
    return SVDLUT_OK;
}

}  // namespace svdlut

using namespace svdlut;

size_t svdlut::backward_workspace(const svdlut_dims *dims, int B, int H, int W, size_t ws_limit)
{
    if (check_dims(dims) != SVDLUT_OK || B < 1 || H < 1 || W < 1) return 0;
    DeviceInfo di;
    if (device_info(&di) != SVDLUT_OK) return 0;
    BwdPlan pl;
    if (plan_backward(dims, B, H, W, di.sm_count, static_cast<size_t>(di.max_smem_optin), ws_limit, &pl) != SVDLUT_OK)
        return 0;
    return pl.total;
}

extern "C" size_t svdlut_backward_workspace_size(const svdlut_dims *dims, int B, int H, int W)
{
    return backward_workspace(dims, B, H, W, SIZE_MAX);
}

extern "C" svdlut_status svdlut_backward(const svdlut_dims *dims, const svdlut_params *params, int B, int H,
                                         int W, const float *x, const float *dy, float *dx,
                                         const svdlut_grads *grads, void *ws, size_t ws_bytes,
                                         svdlut_stream_t stream)
{
    SVDLUT_TRACE("svdlut_backward");
    return backward_limited(dims, params, B, H, W, x, dy, dx, grads, ws, ws_bytes, SIZE_MAX, stream);
}

svdlut_status svdlut::backward_limited(const svdlut_dims *dims, const svdlut_params *params, int B, int H, int W,
                                       const float *x, const float *dy, float *dx, const svdlut_grads *grads,
                                       void *ws, size_t ws_bytes, size_t ws_limit, svdlut_stream_t stream)
{
    clear_error();
    svdlut_status st = check_backward_args(dims, params, B, H, W, x, dy);
    if (st != SVDLUT_OK) return st;
    if (dx && !aligned(dx, 4)) return fail(SVDLUT_ERR_INVALID_ARG, "dx must be 4-byte aligned");
    const size_t img = static_cast<size_t>(3) * H * W * sizeof(float);
    if (dx) {
        const char *ds = reinterpret_cast<const char *>(dx), *xs = reinterpret_cast<const char *>(x),
                   *gs = reinterpret_cast<const char *>(dy);
        const size_t n = B * img;
        if ((ds < xs + n && xs < ds + n) || (ds < gs + n && gs < ds + n))
            return fail(SVDLUT_ERR_INVALID_ARG, "dx overlaps x or dy");
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    DeviceInfo di;
    if ((st = device_info(&di)) != SVDLUT_OK) return st;
    const size_t smem_limit = static_cast<size_t>(di.max_smem_optin);

    const svdlut_grads g0{};
    const svdlut_grads &g = grads ? *grads : g0;
    const bool want_lut = g.dU || g.dS || g.dV || g.dlut_w;
    const bool want_grid = dims->K > 0 && (g.dg_xy || g.dg_xc || g.dg_yc || g.dgrid_w);
    BwdPlan pl;
    if ((st = plan_backward(dims, B, H, W, di.sm_count, smem_limit, ws_limit, &pl)) != SVDLUT_OK) return st;
    const bool have_ws = ws && ws_bytes >= pl.total;
    if ((want_lut || want_grid) && !have_ws)
        return fail(SVDLUT_ERR_WORKSPACE, "workspace of %zu bytes needed (got %zu)", pl.total, ws ? ws_bytes : 0);
    if (have_ws && !aligned(ws, 256)) return fail(SVDLUT_ERR_INVALID_ARG, "workspace must be 256-byte aligned");

    // 1. dx through the forward kernel's adjoint mode, up to 16 images per
    // launch, or 64 when the batch is larger
    if (dx) {
        char *tables = have_ws ? static_cast<char *>(ws) + pl.off_prep : nullptr;
        st = B > kPlainChunk ? dx_chunks<kRaggedMax>(dims, params, B, H, W, x, dy, dx, tables, pl.prep_img, di, s)
                             : dx_chunks<kPlainChunk>(dims, params, B, H, W, x, dy, dx, tables, pl.prep_img, di, s);
        if (st != SVDLUT_OK) return st;
    }
    if (!want_lut && !want_grid) return SVDLUT_OK;
    char *w = static_cast<char *>(ws);
    float *lut_part = reinterpret_cast<float *>(w + pl.off_lut);
    float *sums_part = reinterpret_cast<float *>(w + pl.off_sums);
    float *grid_part = reinterpret_cast<float *>(w + pl.off_grid);
    float *wpart = reinterpret_cast<float *>(w + pl.off_wpart);

    BwdArgs a{};
    a.x = x;
    a.dy = dy;
    a.B = B;
    a.H = H;
    a.W = W;
    a.D = dims->D_t;
    a.K = dims->K;
    a.Dsx = dims->Dsx;
    a.Dsy = dims->Dsy;
    a.Dsc = dims->Dsc;
    a.rW1 = W > 1 ? 1.0f / static_cast<float>(W - 1) : 0.f;
    a.rH1 = H > 1 ? 1.0f / static_cast<float>(H - 1) : 0.f;
    a.strips = (W + kTileW - 1) / kTileW;
    a.vec = (W % 4 == 0) && aligned(x, 16) && aligned(dy, 16);
    a.seg = lut_segment(pl.G, B);

    if ((st = allow_dynamic_smem(reinterpret_cast<const void *>(lut_grad_kernel), di.max_smem_optin, di.device)) !=
        SVDLUT_OK)
        return st;
    if ((st = allow_dynamic_smem(reinterpret_cast<const void *>(grid_grad_kernel), di.max_smem_optin, di.device)) !=
        SVDLUT_OK)
        return st;
    if ((st = allow_dynamic_smem(reinterpret_cast<const void *>(lut_finalize_kernel), di.max_smem_optin,
                                 di.device)) != SVDLUT_OK)
        return st;
    if (pl.grid_smem + 256 > static_cast<size_t>(di.max_smem_optin) || pl.lut_smem > static_cast<size_t>(di.max_smem_optin))
        return fail(SVDLUT_ERR_UNSUPPORTED, "adjoint tables do not fit in shared memory");
    // 2. LUT pass (also produces the dy channel sums used by every bias)
    if ((st = launch_pdl(lut_grad_kernel, dim3(pl.G), dim3(kLutThreads), pl.lut_smem, s, a, lut_part, sums_part)) !=
        SVDLUT_OK)
        return st;
    if (want_lut) {
        FinArgs f{params->U, params->S, params->V, params->lut_w, g.dU, g.dS, g.dV, g.dlut_w,
                  dims->D_t, dims->rank, B, pl.G, a.seg, pl.units};
        const size_t fsm = sizeof(float) * fin_smem_floats(dims->D_t, dims->rank);
        if ((st = launch_pdl(lut_finalize_kernel, dim3(9, B), dim3(9 * B <= di.sm_count ? kFinMaxThreads : kFinMaxThreads / 2), fsm, s, f,
                             static_cast<const float *>(lut_part), static_cast<const float *>(sums_part))) != SVDLUT_OK)
            return st;
    }
    if (want_grid) {
        if ((st = launch_pdl(grid_grad_kernel, dim3(pl.gp.nblk, B), dim3(pl.gp.groups * 3 * 32), pl.grid_smem, s, a,
                             pl.gp, grid_part)) != SVDLUT_OK)
            return st;
        GridRed r{};
        r.B = B;
        r.H = H;
        r.W = W;
        r.K = dims->K;
        r.Dsx = dims->Dsx;
        r.Dsy = dims->Dsy;
        r.Dsc = dims->Dsc;
        r.strips = a.strips;
        r.rW1 = a.rW1;
        r.rH1 = a.rH1;
        r.gp = pl.gp;
        r.smax = pl.smax;
        for (int q = 0; q < 3; ++q) r.sl[q] = pl.sl[q];
        r.gxy = params->g_xy;
        r.gxc = params->g_xc;
        r.gyc = params->g_yc;
        r.gw = params->grid_w;
        r.dgxy = g.dg_xy;
        r.dgxc = g.dg_xc;
        r.dgyc = g.dg_yc;
        r.wpart = g.dgrid_w ? wpart : nullptr;
        // the CTA's band and strip footprint tables, then its warps' sums
        const size_t rsm = std::max(sizeof(int) * 2 * static_cast<size_t>(pl.gp.bands + a.strips),
                                    sizeof(float) * (kGRThreads / 32) * dims->K);
        if (rsm > 48 * 1024) {
            if ((st = allow_dynamic_smem(reinterpret_cast<const void *>(grid_reduce_kernel), di.max_smem_optin,
                                         di.device)) != SVDLUT_OK)
                return st;
            if (rsm > static_cast<size_t>(di.max_smem_optin))
                return fail(SVDLUT_ERR_UNSUPPORTED, "too many column strips and row bands for the grid reduction");
        }
        if ((st = launch_pdl(grid_reduce_kernel, dim3(pl.sl[0] + pl.sl[1] + pl.sl[2], B), dim3(kGRThreads), rsm, s,
                             r, static_cast<const float *>(grid_part))) != SVDLUT_OK)
            return st;
        if (g.dgrid_w) {
            GridWsum f{B, dims->K, pl.G, a.seg, pl.smax, {pl.sl[0], pl.sl[1], pl.sl[2]}, g.dgrid_w, pl.units};
            const int n = B * dims->K * 4;
            if ((st = launch_pdl(grid_wsum_kernel, dim3((n + 255) / 256), dim3(256), 0, s, f,
                                 static_cast<const float *>(wpart), static_cast<const float *>(sums_part))) != SVDLUT_OK)
                return st;
        }
    }
    return SVDLUT_OK;
}
