// Coefficients of the FP64 depth march (csrc/green.cu), read by its evaluations and by the
// reverse-mode gradients.
#pragma once
#include "edt_internal.h"
#include "cplx.cuh"

namespace edt {

// coefficient slots per (f, n, layer): kappa; sigma, then M; tau, then T; exp(i kappa dz),
// exp(-i kappa dz); exp(i kappa h); delta, then D (see green_layer and green_recursion)
constexpr int NCOEF = 7;
constexpr int C_KAP = 0, C_SIG = 1, C_MUP = 1, C_AMP = 2, C_E = 3, C_EI = 4, C_EH = 5, C_DEL = 6, C_DEN = 6;
// coefficient array layout [f][layer][slot][n]: consecutive wavenumbers are adjacent, so the
// per-(f, n) threads of every kernel below read and write them coalesced
__device__ __forceinline__ size_t cix(const Dev& d, int f, int n, int j, int k) {
  return ((size_t(f) * d.nlayer + j) * NCOEF + k) * d.nk + n;
}

// 1 / b with one real division (|b| is O(1e-3 .. 1e3) for every use here)
__device__ __forceinline__ double2 cinv(double2 b) {
  const double r = 1.0 / (b.x * b.x + b.y * b.y);
  return cmk(b.x * r, -b.y * r);
}

// amplitude and reflection of layer j from the recursion's M, D, T
__device__ __forceinline__ void layer_waves(const Dev& d, int f, int n, int j, double2& amp, double2& rho) {
  const double2 D = d.coef[cix(d, f, n, j, C_DEN)];
  amp = d.coef[cix(d, f, n, j, C_AMP)] * D;
  rho = j < d.nlayer - 1 ? d.coef[cix(d, f, n, j, C_MUP)] * cinv(D) : cmk(0.0, 0.0);
}

// the same with kappa_j and exp(i kappa_j h_j)
struct GreenLayer { double2 kappa, eh, amp, rho; };
__device__ __forceinline__ double2 green_layer_eh(const Dev& d, int f, int n, int j) {
  return d.coef[cix(d, f, n, j, C_EH)];
}
__device__ __forceinline__ GreenLayer green_layer_state(const Dev& d, int f, int n, int j) {
  GreenLayer q;
  q.kappa = d.coef[cix(d, f, n, j, C_KAP)];
  q.eh = j < d.nlayer - 1 ? green_layer_eh(d, f, n, j) : cmk(1.0, 0.0);
  layer_waves(d, f, n, j, q.amp, q.rho);
  return q;
}

}  // namespace edt
