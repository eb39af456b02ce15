// The instances of apply_kernel: included by the translation units that
// instantiate launch_io, one (format, N, direction) each, so that they compile
// in parallel and once.
#pragma once

#include "apply_kernel.cuh"
#include "apply_launch.cuh"

namespace svdlut {

// Launches one instance as a dependent of the preceding kernel (prep_kernel, or
// any other): it may be launched while that one runs, and waits for it before
// it reads anything (after prep_kernel, before it reads the tables: prep_kernel
// has waited for what came before).
template <class IO, int N, bool DX, int PRE, bool FAST, bool VEC>
svdlut_status launch_instance_v(LaunchArgs<N> &a, size_t smem, const DeviceInfo &di, cudaStream_t s, int grid)
{
    svdlut_status st = allow_smem_once(reinterpret_cast<const void *>(apply_kernel<IO, N, DX, PRE, FAST, VEC>),
                                       di.max_smem_optin, di.device);
    if (st != SVDLUT_OK) return st;
    if ((st = check_buffer(&a.check)) != SVDLUT_OK) return st;
    if (grid <= 0) grid = std::min(a.total_blocks, di.sm_count);
    grid = std::max(1, std::min(grid, a.total_blocks));
    return launch_pdl(apply_kernel<IO, N, DX, PRE, FAST, VEC>, dim3(grid), dim3(kThreads), smem, s, a);
}

// Float images take the aligned instance where every image is aligned.
template <class IO, int N, bool DX, int PRE, bool FAST>
svdlut_status launch_instance(LaunchArgs<N> &a, size_t smem, const DeviceInfo &di, cudaStream_t s, int grid)
{
    if constexpr (std::is_same<IO, IoF32>::value && (FAST || DX)) {
        bool vec = true;
        for (int i = 0; i < a.n; ++i) vec = vec && a.img[i].vec;
        if (vec) return launch_instance_v<IO, N, DX, PRE, FAST, true>(a, smem, di, s, grid);
    }
    return launch_instance_v<IO, N, DX, PRE, FAST, false>(a, smem, di, s, grid);
}

template <class IO, int N, bool DX>
svdlut_status launch_io(LaunchArgs<N> &a, size_t smem, const DeviceInfo &di, cudaStream_t s, int grid)
{
    if constexpr (!DX)
        if (a.pre == kPreFolds) return launch_instance<IO, N, DX, kPreFolds, true>(a, smem, di, s, grid);
    const bool fast = all_fast_rows(a);
    if constexpr (std::is_same<IO, IoF32>::value && !DX)  // 1 % at most; none with 8-bit pixels
        if (a.pre && fast) return launch_instance<IO, N, DX, kPreAll, true>(a, smem, di, s, grid);
    if (a.pre) return launch_instance<IO, N, DX, kPreAll, false>(a, smem, di, s, grid);
    return fast ? launch_instance<IO, N, DX, kPreNone, true>(a, smem, di, s, grid)
                : launch_instance<IO, N, DX, kPreNone, false>(a, smem, di, s, grid);
}

}  // namespace svdlut
