// apply_kernel for the transform of 8-bit planar images, up to 64 per launch.
#include "apply_instances.cuh"

template svdlut_status svdlut::launch_io<svdlut::IoU8, 64, false>(svdlut::LaunchArgs<64> &, size_t,
                                                            const svdlut::DeviceInfo &, cudaStream_t, int);
