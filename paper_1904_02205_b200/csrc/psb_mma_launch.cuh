// Launch of one K-block instance of the contraction kernel; included by the translation units that instantiate it.
#pragma once

#include "psb_mma.cuh"

namespace psb {

template <int BK>
cudaError_t launch_mma_kernel(const cudaLaunchConfig_t& cfg, const TmapSet& maps, const TensorParams& p, int device, int kind) {
  const auto kernel = kind == kGeneralOutputs ? psb_mma_kernel<BK, kGeneralOutputs>
                      : kind == kRealOutputs  ? psb_mma_kernel<BK, kRealOutputs>
                      : kind == kSortedRows   ? psb_mma_kernel<BK, kSortedRows> : psb_mma_kernel<BK, kOneLevel>;
  // the shared-memory limit of an instance is raised once per device, to the most a launch can ask for
  constexpr int kMaxDevicesForAttr = 64;
  static bool raised[kMaxDevicesForAttr][4];
  const bool known = device >= 0 && device < kMaxDevicesForAttr;
  if (!known || !raised[device][kind]) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget);
    if (e != cudaSuccess) return e;
    if (known) raised[device][kind] = true;
  }
  return cudaLaunchKernelEx(&cfg, kernel, maps, p);
}

}  // namespace psb
