// Launch of one K-block instance of the contraction kernel; included by the translation units that instantiate it.
#pragma once

#include "psb_mma.cuh"

namespace psb {

template <int BK>
cudaError_t launch_mma_kernel(const cudaLaunchConfig_t& cfg, const TmapSet& maps, const TensorParams& p, int device, bool general) {
  // the shared-memory limit of an instance is raised once per device, to the most a launch can ask for
  constexpr int kMaxDevicesForAttr = 64;
  static bool raised[kMaxDevicesForAttr][2];
  const bool known = device >= 0 && device < kMaxDevicesForAttr;
  if (!known || !raised[device][general]) {
    const cudaError_t e = general
        ? cudaFuncSetAttribute(psb_mma_kernel<BK, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget)
        : cudaFuncSetAttribute(psb_mma_kernel<BK, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget);
    if (e != cudaSuccess) return e;
    if (known) raised[device][general] = true;
  }
  return general ? cudaLaunchKernelEx(&cfg, psb_mma_kernel<BK, true>, maps, p)
                 : cudaLaunchKernelEx(&cfg, psb_mma_kernel<BK, false>, maps, p);
}

}  // namespace psb
