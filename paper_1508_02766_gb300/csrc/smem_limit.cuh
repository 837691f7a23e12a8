// The dynamic shared memory limit of a kernel, raised to all that the device
// gives a block (the opt-in limit covers static and dynamic together).
#pragma once

#include <cuda_runtime.h>

#include "device_once.h"

namespace kde {

constexpr size_t kSmemMax = 227 * 1024;

template <typename F>
cudaError_t allow_smem(F* fn) {
  static DeviceOnce once;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  return once.run<cudaError_t>(dev, (const void*)fn, [&] {
    cudaFuncAttributes attr{};
    const cudaError_t e1 = cudaFuncGetAttributes(&attr, fn);
    if (e1 != cudaSuccess) return e1;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kSmemMax - attr.sharedSizeBytes));
  });
}

}  // namespace kde
