// Eq. 2's pointwise functions where a convolution kernel applies them as it reads its tensors.
#pragma once
#include "common.cuh"

namespace hn {

__device__ __forceinline__ float mix_sigmoid(float x) { return 1.f / (1.f + __expf(-x)); }

// element type a kernel writes: fp32 where the operator's outer RMSNorm follows
template <typename T, bool MIX> struct MixOut { using type = T; };
template <typename T> struct MixOut<T, true> { using type = float; };

}  // namespace hn
