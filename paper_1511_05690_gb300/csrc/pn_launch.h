// Host helpers of the kernel launches.
#pragma once
#include <cuda_runtime.h>

#include "pn_split.h"

namespace pn {

// Lets Kernel take up to `bytes` of dynamic shared memory (always the same figure for
// one kernel: its largest, so that no thread lowers it under another's launch).
// The attribute belongs to the current device and is set once on each.
template <auto Kernel>
inline cudaError_t allow_smem(int bytes) {
  static DeviceSet done;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || done.has(dev)) return e;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.add(dev);
  return e;
}

}  // namespace pn
