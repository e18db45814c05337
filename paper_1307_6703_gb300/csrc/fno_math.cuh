// fno_math.cuh -- the network's activation, shared by its kernels.
#pragma once

#include <cuda_runtime.h>

namespace fno {

// gelu(z) = z Phi(z), Phi the standard normal distribution function.
__device__ __forceinline__ float gelu(float z) { return z * normcdff(z); }
__device__ __forceinline__ float gelu_grad(float z) {
  return normcdff(z) + z * (0.3989422804014327f * expf(-0.5f * z * z));
}

}  // namespace fno
