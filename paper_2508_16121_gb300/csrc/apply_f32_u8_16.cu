// apply_kernel for float -> 8-bit planar images, up to 16 per launch.
#include "apply_instances.cuh"

template svdlut_status svdlut::launch_io<svdlut::Io<svdlut::InF32, svdlut::OutU8>, 16, false>(
    svdlut::LaunchArgs<16> &, size_t, const svdlut::DeviceInfo &, cudaStream_t, int);
