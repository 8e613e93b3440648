// The contraction kernel (psb_mma.cuh) for K blocks of 64 bytes.
#include "psb_mma_launch.cuh"

namespace psb {
template cudaError_t launch_mma_kernel<64>(const cudaLaunchConfig_t&, const TmapSet&, const TensorParams&, int, int, int);
}  // namespace psb
