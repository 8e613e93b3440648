// Launch of one K-block instance of the contraction kernel; included by the translation units that instantiate it.
#pragma once

#include "psb_mma.cuh"

namespace psb {

template <int BK>
cudaError_t launch_mma_kernel(const cudaLaunchConfig_t& cfg, const TmapSet& maps, const TensorParams& p, int device, int kind, int rec) {
  typedef void (*Kernel)(const TmapSet, const TensorParams);
  static const Kernel kernels[5][3] = {
      {psb_mma_kernel<BK, kOneLevel, kPlainSums>, psb_mma_kernel<BK, kOneLevel, kMidSums>, psb_mma_kernel<BK, kOneLevel, kAddSums>},
      {psb_mma_kernel<BK, kSortedRows, kPlainSums>, psb_mma_kernel<BK, kSortedRows, kMidSums>, psb_mma_kernel<BK, kSortedRows, kAddSums>},
      {psb_mma_kernel<BK, kGeneralOutputs, kPlainSums>, nullptr, nullptr},
      {psb_mma_kernel<BK, kRealOutputs, kPlainSums>, nullptr, nullptr},
      {psb_mma_kernel<BK, kRealSorted, kPlainSums>, nullptr, nullptr}};
  const Kernel kernel = kernels[kind][rec];
  // the shared-memory limit of an instance is raised once per device, to the most a launch can ask for
  constexpr int kMaxDevicesForAttr = 64;
  static bool raised[kMaxDevicesForAttr][5][3];
  const bool known = device >= 0 && device < kMaxDevicesForAttr;
  if (!known || !raised[device][kind][rec]) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget);
    if (e != cudaSuccess) return e;
    if (known) raised[device][kind][rec] = true;
  }
  return cudaLaunchKernelEx(&cfg, kernel, maps, p);
}

}  // namespace psb
