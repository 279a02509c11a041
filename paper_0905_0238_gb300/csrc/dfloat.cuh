// Double-float arithmetic on the FP32 pipes: a value is the unevaluated sum h + l of two floats
// (float2: .x high part, .y low part, about 48 significant bits).  Products are split exactly by
// fma (Dekker's TwoProduct with a hardware fma), additions' rounding errors captured by Knuth's
// TwoSum; the _rn intrinsics keep the compiler from contracting the error-free steps into fma.
// Shared by the double-float Cholesky of the line path and the trailing updates of the
// streaming path's blocked Cholesky.
#pragma once
#include <cuda_runtime.h>

namespace edt {

__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ float2 fast_two_sum(float a, float b) {   // |a| >= |b| or a == 0
  const float s = __fadd_rn(a, b);
  return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ float2 df_norm(float2 a) { return fast_two_sum(a.x, a.y); }
__device__ __forceinline__ float2 df_of(double x) {
  const float h = __double2float_rn(x);
  return make_float2(h, __double2float_rn(x - double(h)));
}
__device__ __forceinline__ double df_val(float2 a) { return double(a.x) + double(a.y); }
__device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
  const float2 s = two_sum(a.x, b.x);
  return fast_two_sum(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = fmaf(a.x, b.y, fmaf(a.y, b.x, fmaf(a.x, b.x, -p)));
  return fast_two_sum(p, e);
}
// accumulator s (high sum, low sum; not normalised) += a * b
__device__ __forceinline__ void df_acc(float2& s, float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = fmaf(a.x, b.y, fmaf(a.y, b.x, fmaf(a.x, b.x, -p)));
  const float2 t = two_sum(s.x, p);
  s.x = t.x;
  s.y = __fadd_rn(s.y, __fadd_rn(t.y, e));
}
__device__ __forceinline__ float2 shfl_df(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// exact product of two hi parts split as (rounded product, its error)
__device__ __forceinline__ float two_prod_err(float a, float b, float p) { return fmaf(a, b, -p); }

// a_h + a_l = (ph + pl)(qh + ql) for one complex depth value, to ~2^-44 relative
__device__ __forceinline__ void cmul_df(float2 ph, float2 pl, float2 qh, float2 ql, float2& ah, float2& al) {
  const float p1 = __fmul_rn(ph.x, qh.x), p2 = __fmul_rn(ph.y, qh.y);
  const float e1 = two_prod_err(ph.x, qh.x, p1), e2 = two_prod_err(ph.y, qh.y, p2);
  const float sr = __fsub_rn(p1, p2);
  const float br = __fsub_rn(sr, p1);
  const float er = __fadd_rn(__fsub_rn(p1, __fsub_rn(sr, br)), __fsub_rn(-p2, br));
  const float cr = fmaf(ph.x, ql.x, fmaf(pl.x, qh.x, -fmaf(ph.y, ql.y, __fmul_rn(pl.y, qh.y))));
  const float p3 = __fmul_rn(ph.x, qh.y), p4 = __fmul_rn(ph.y, qh.x);
  const float e3 = two_prod_err(ph.x, qh.y, p3), e4 = two_prod_err(ph.y, qh.x, p4);
  const float si = __fadd_rn(p3, p4);
  const float bi = __fsub_rn(si, p3);
  const float ei = __fadd_rn(__fsub_rn(p3, __fsub_rn(si, bi)), __fsub_rn(p4, bi));
  const float ci = fmaf(ph.x, ql.y, fmaf(pl.x, qh.y, fmaf(ph.y, ql.x, __fmul_rn(pl.y, qh.x))));
  ah = make_float2(sr, si);
  al = make_float2(((e1 - e2) + er) + cr, ((e3 + e4) + ei) + ci);
}

// 1 / sqrt(a) for a double-float a > 0: the FP32 estimate y0 and one Newton step,
// y = y0 - y0 e / 2 with e = a y0^2 - 1 formed by fused multiply-adds on the exact square
// y0^2 = ph + pl (each fma rounds a quantity of order 2^-22 once, so e carries ~2^-46 absolute
// error); the step doubles the ~23 correct bits of the estimate.  Nine dependent operations
// after the estimate, on the critical path of every pivot.
__device__ __forceinline__ float2 df_rsqrt(float2 a) {
  const float y0 = rsqrtf(a.x);
  const float ph = __fmul_rn(y0, y0);
  const float pl = fmaf(y0, y0, -ph);
  float e = fmaf(a.x, ph, -1.0f);
  e = fmaf(a.x, pl, e);
  e = fmaf(a.y, ph, e);
  return fast_two_sum(y0, __fmul_rn(__fmul_rn(-0.5f, y0), e));
}

// ---- one 32 x 32 diagonal block of a blocked double-float Cholesky factorisation ----------
// Shared scratch of the diagonal-block factorisation.
struct DfDiagScratch {
  float2 col[32][33];                             // the block, then L, by columns
  float2 ls[3][32];                               // column j of L over L_jj (three in use at a time)
  float2 xr[2][32];                               // finished rows of U (below)
  float2 inv[32];                                 // 1 / L_jj
  int fail;                                       // a pivot failed; read after the last column only
};

// Diagonal block of step k0 of one subproblem (kb = min(32, n - k0) columns), factored and
// inverted in double-float by a 256-thread CTA; lane i of a warp holds row i of the columns
// c = warp + 8 q, q < 4.  Right-looking with a one-column look-ahead, one barrier per column: in the
// phase that subtracts column j from the trailing block, the warp of column j + 1, which that
// subtraction finishes, takes its pivot from its own lane j + 1 and scales the column, which is
// ready at the next barrier.  A finished column's registers go on to hold its column of U, L^-1 = X
// with X_ic = U_ic / L_ii: U_i = e_i - sum_{k < i} (L_ik / L_kk) U_k, updated in the same phases
// with row j - 1.  So a warp does one product per column it holds and phase; A's entries and U's in separate
// registers, with a lane per column, took two, and the scaling ran in every warp with one lane (the
// first blocks of the 2050 systems of a 64 x 64 grid: 149 us then, 107 now; its inversion 2.36 ms, 2.23).
// Writes L_kk (lower triangle) and its FP32 copy (L32, may be null; X goes there too), X to the strict
// upper triangle (X_il at (l, i)), and the reciprocal pivots (dinv FP64; dinv32 FP32, may be null).  A
// non-positive or non-finite pivot sets EDT_ENOTPD and returns false (in every thread), after all columns:
// a thread that left the loop by itself would miss barriers that the others wait at, and what follows a
// failed pivot is not written.  Every thread of the CTA calls it; A's block must be final and visible to the CTA.
__device__ inline bool df_diag_block(float2* A, float* L32, double* dinv, float* dinv32, int* status, int n,
                                     int k0, DfDiagScratch& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kb = min(32, n - k0);
  const float2 zero = make_float2(0.f, 0.f), one = make_float2(1.f, 0.f);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = warp + 8 * q;
    sh.col[lane][i] = i < kb && lane <= i ? A[size_t(k0 + i) * n + k0 + lane] : zero;
  }
  if (threadIdx.x == 0) sh.fail = 0;
  if (threadIdx.x < 64) sh.xr[threadIdx.x >> 5][lane] = zero;
  if (threadIdx.x < 96) sh.ls[threadIdx.x >> 5][lane] = zero;
  __syncthreads();
  float2 w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = sh.col[warp + 8 * q][lane];
  // column j from its finished entries v, by the warp that holds it
  auto column = [&](int j, float2& v) {
    const float2 d = df_norm(shfl_df(v, j));
    if ((!(d.x > 0.f) || !isfinite(d.x)) && lane == 0) sh.fail = 1;
    const float2 iv = df_rsqrt(d);
    const float2 l = df_mul(lane == j ? d : df_norm(v), iv);
    if (lane >= j) {
      sh.col[j][lane] = l;
      sh.ls[j % 3][lane] = df_mul(l, iv);
    }
    if (lane == 0) sh.inv[j] = iv;
    v = lane == j ? one : zero;                   // from here on the column of U
  };
  if (warp == 0) column(0, w[0]);
  __syncthreads();
  for (int j = 0; j < kb; ++j) {
    // columns c > j: A -= L_j L_j^T (rows above c are not used); c < j: U_i -= (L_i,j-1 / L_j-1,j-1) U_j-1
    // for the rows i >= j, the others and column j subtract zero
    const float2 lj = df_neg(sh.col[j][lane]);
    const float2 lp = lane >= j ? df_neg(sh.ls[(j + 2) % 3][lane]) : zero;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = warp + 8 * q;                 // the same in the whole warp
      const float2 o = c > j ? sh.col[j][c] : sh.xr[(j + 1) & 1][c];
      df_acc(w[q], c > j ? lj : c < j ? lp : zero, o);
    }
    if (lane == j) {                              // row j of U
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (warp + 8 * q <= j) sh.xr[j & 1][warp + 8 * q] = df_norm(w[q]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (j + 1 < kb && warp + 8 * q == j + 1) column(j + 1, w[q]);
    __syncthreads();
  }
  if (sh.fail) {                                  // not written since the last barrier
    if (threadIdx.x == 0) *status = EDT_ENOTPD;
    return false;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = warp + 8 * q;                   // L row i, column lane
    if (i < kb && lane <= i) {
      const float2 l = sh.col[lane][i];
      A[size_t(k0 + i) * n + k0 + lane] = l;
      if (L32) L32[size_t(k0 + i) * n + k0 + lane] = l.x;
    }
    if (lane < kb && i < lane) {                  // X_{lane, i} to the upper triangle
      const float2 x = df_mul(df_norm(w[q]), sh.inv[lane]);
      A[size_t(k0 + i) * n + k0 + lane] = x;
      if (L32) L32[size_t(k0 + i) * n + k0 + lane] = x.x;
    }
  }
  if (threadIdx.x < kb) {
    dinv[k0 + threadIdx.x] = df_val(sh.inv[threadIdx.x]);
    if (dinv32) dinv32[k0 + threadIdx.x] = sh.inv[threadIdx.x].x;
  }
  return true;
}
}  // namespace edt
