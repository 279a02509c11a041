// Reductions of several values over a warp together.
#pragma once
#include <cuda_runtime.h>

namespace edt {

// K values (a power of two below 32) reduced over the warp by op: each exchange halves the values a
// lane carries, so K - 1 + 5 - log2 K shuffles do what one butterfly per value does in 5 K.  Lane l
// returns value l >> (5 - log2 K), its operands paired as a butterfly over spans 16, 8, 4, 2, 1
// pairs them.
template <int K, class Op>
__device__ __forceinline__ float warp_fold(float (&v)[K], int lane, const Op& op) {
  int span = 16;
#pragma unroll
  for (int k = K / 2; k >= 1; k >>= 1, span >>= 1) {
    const bool hi = lane & span;
#pragma unroll
    for (int j = 0; j < k; ++j) {
      const float give = hi ? v[j] : v[j + k], keep = hi ? v[j + k] : v[j];
      v[j] = op(keep, __shfl_xor_sync(0xffffffffu, give, span));
    }
  }
#pragma unroll
  for (; span > 0; span >>= 1) v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], span));
  return v[0];
}

template <int K>
__device__ __forceinline__ float warp_sums(float (&v)[K], int lane) {
  return warp_fold(v, lane, [](float a, float b) { return a + b; });
}

}  // namespace edt
