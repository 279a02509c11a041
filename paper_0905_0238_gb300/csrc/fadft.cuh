// Small in-register DFTs shared by the window geometry's transforms (csrc/fa.cu, csrc/fagrid.cu).
#pragma once
#include "cplx.cuh"
#include "wfft.cuh"

namespace edt {

// cos and sin of 2 pi k / 16
__device__ __forceinline__ float2 w16(int k) {
  constexpr float C[16] = {1.f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
                           0.f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f,
                           -1.f, -0.92387953251128674f, -0.70710678118654752f, -0.38268343236508977f,
                           0.f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f};
  return make_float2(C[k & 15], -C[(k + 12) & 15]);        // e^{-2 pi i k/16} = (cos, -sin)
}

// In-register DFTs of R points with either sign (natural order)
template <int R, int SG> struct Dft;
template <int SG> struct Dft<2, SG> {
  __device__ static __forceinline__ void run(float2 (&a)[2]) {
    const float2 u = a[0], v = a[1];
    a[0] = u + v; a[1] = u - v;
  }
};
template <int SG> struct Dft<4, SG> {
  __device__ static __forceinline__ void run(float2 (&a)[4]) {
    const float2 b0 = a[0] + a[2], b1 = a[0] - a[2], b2 = a[1] + a[3], b3 = rot4<SG>(a[1] - a[3]);
    a[0] = b0 + b2; a[2] = b0 - b2; a[1] = b1 + b3; a[3] = b1 - b3;
  }
};
template <int SG> struct Dft<8, SG> {
  __device__ static __forceinline__ void run(float2 (&a)[8]) { dft8<SG>(a); }
};
template <int SG> struct Dft<16, SG> {
  __device__ static __forceinline__ void run(float2 (&a)[16]) {
    float2 e[8], o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { e[i] = a[2 * i]; o[i] = a[2 * i + 1]; }
    dft8<SG>(e);
    dft8<SG>(o);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float2 t = o[k] * tw_sg<SG>(w16(k));
      a[k] = e[k] + t;
      a[k + 8] = e[k] - t;
    }
  }
};

}  // namespace edt
