// nn_device.cuh -- device helpers shared by the network kernels.
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

#include "nn_internal.h"

namespace mach_nn {

// Two rounded bfloat16 gradients times the leaky ReLU's derivative at activations m (the
// product with a power of two rounds as scaling the stored gradient would).
__device__ __forceinline__ uint32_t lrelu_grad2(uint32_t g, uint32_t m) {
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&m));
  const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&g));
  const __nv_bfloat162 b = __floats2bfloat162_rn(a.x > 0.f ? v.x : v.x * kLeak, a.y > 0.f ? v.y : v.y * kLeak);
  return *reinterpret_cast<const uint32_t*>(&b);
}
__device__ __forceinline__ uint4 lrelu_grad8(uint4 g, uint4 m) {
  return make_uint4(lrelu_grad2(g.x, m.x), lrelu_grad2(g.y, m.y), lrelu_grad2(g.z, m.z), lrelu_grad2(g.w, m.w));
}

}  // namespace mach_nn
