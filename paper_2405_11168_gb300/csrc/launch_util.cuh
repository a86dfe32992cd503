// Launch helpers shared by the kernel units.
#pragma once
#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <utility>

#include "launch.h"

namespace hs {

// Raise a kernel's dynamic shared-memory limit when a launch needs more than
// it has been given so far on the current device (the attribute is per device,
// so the record is keyed by device ordinal and kernel).  Launches recorded into
// a graph capture therefore never call the attribute API: the first,
// uncaptured, chunk of a solve has already set it.
inline std::mutex& smem_mu() {
  static std::mutex m;
  return m;
}
inline std::map<std::pair<int, const void*>, size_t>& smem_set() {
  static std::map<std::pair<int, const void*>, size_t> m;
  return m;
}
template <typename K> static cudaError_t set_smem(K kernel, size_t smem) {
  if (smem <= 48 * 1024) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const std::pair<int, const void*> key(dev, reinterpret_cast<const void*>(kernel));
  std::lock_guard<std::mutex> lock(smem_mu());
  size_t& have = smem_set()[key];
  if (smem <= have) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) have = smem;
  return e;
}

// Launch of a transform pass, plainly or as a programmatic dependent of the kernel before it.
template <typename K, typename A>
static cudaError_t launch_pass(K kernel, const A& a, bool dependent, dim3 g, int nthr, size_t smem, cudaStream_t s) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = g;
  cfg.blockDim = dim3((unsigned)nthr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

}  // namespace hs
