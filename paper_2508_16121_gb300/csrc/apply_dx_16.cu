// apply_kernel for the adjoint of the transform of float images, up to 16 per launch.
#include "apply_instances.cuh"

template svdlut_status svdlut::launch_io<svdlut::IoF32, 16, true>(svdlut::LaunchArgs<16> &, size_t,
                                                            const svdlut::DeviceInfo &, cudaStream_t, int);
