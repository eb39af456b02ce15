// apply_kernel for interleaved 8-bit -> interleaved 8-bit images, up to 16 per launch.
#include "apply_instances.cuh"

template svdlut_status svdlut::launch_io<svdlut::Io<svdlut::InU8Hwc, svdlut::OutU8Hwc>, 16, false>(
    svdlut::LaunchArgs<16> &, size_t, const svdlut::DeviceInfo &, cudaStream_t, int);
