// Substitutions L L^T x = b with a blocked Cholesky factor whose 32 x 32 diagonal blocks carry
// their inverses, for two right-hand sides at once, by one CTA.
//
// Layout of the factor: L lower, row-major with leading dimension n; the strict upper triangle
// of each diagonal block holds X = L_kk^-1 (X_il at (l, i)); the diagonal of X (1 / L_ii) is
// passed separately.  Every load of the factor is coalesced: lanes run across one row's 32
// columns of a block, warps across rows, and each warp keeps 16 row segments loading at once
// (the factor is usually read from DRAM, and one CTA per system must cover the latency with
// loads in flight).  Each block is one barrier-separated pass:
//   forward   t = b_blk - L[blk, 0:k0] y[0:k0]: one warp per row, lanes over the columns, a
//             shuffle butterfly for the dot product; then y_blk = X t (warp r: right-hand side r,
//             lane: row);
//   backward  t = y_blk - L[k0+kb:n, blk]^T x[k0+kb:n]: lane = column, warps over the rows,
//             the warps' partial sums added in warp order; then x_blk = X^T t.
// Every sum runs in a fixed order, so the result is bitwise reproducible.  Two arithmetic
// forms: double-float (float2 pairs, the factorisation's working precision) and FP32 (the
// refinement's correction solves with the factor's FP32 copy).
#pragma once
#include "dfloat.cuh"

namespace edt {

struct DfArith {
  using T = float2;
  static __device__ __forceinline__ T zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ void acc(T& s, T a, T b) { df_acc(s, a, b); }
  static __device__ __forceinline__ T add(T a, T b) { return df_add(a, b); }
  static __device__ __forceinline__ T sub(T a, T b) { return df_add(a, df_neg(b)); }
  static __device__ __forceinline__ T norm(T a) { return df_norm(a); }
  // the xor butterfly gives every lane the same sum: TwoSum's error term does not depend on
  // the order of its operands
  static __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      v = df_add(v, make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o)));
    return v;
  }
};

struct F32Arith {
  using T = float;
  static __device__ __forceinline__ T zero() { return 0.f; }
  static __device__ __forceinline__ void acc(T& s, T a, T b) { s = fmaf(a, b, s); }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ T sub(T a, T b) { return a - b; }
  static __device__ __forceinline__ T norm(T a) { return a; }
  static __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
};

constexpr int BS_B = 32, BS_LD = 33;

// Shared scratch (elements of Ar::T): sX [32 * 33], red [NT / 32 * 2 * 32].
template <class Ar, int NT>
__host__ __device__ constexpr int blk_solve_scratch() { return BS_B * BS_LD + NT / 32 * 2 * BS_B; }

// Solves L L^T x = b in place: sb[i][r] (shared, [n][2]) holds b on entry and x on return.
// inv_diag: 1 / L_ii ([n], shared or global).  Called by all NT threads of the CTA.
//
// A block's loads do not depend on the solution, so the next block's inverse and its first column
// chunks (or rows, backward) are requested before this block's reductions and barriers, and
// within a block the next chunk before this one is used: one CTA per system is bound by these
// latencies.  With the panels' side-by-side sums (csrc/chol_df.cu, csrc/chol.cu) an inversion of a
// 256-point line with 150 depths takes 1.114 ms against 1.127, a burst of 32 requests 2.11 against 2.19.
template <class Ar, int NT>
__device__ void blk_solve_2rhs(const typename Ar::T* A, const typename Ar::T* inv_diag, int n,
                               typename Ar::T* sb, typename Ar::T* scratch) {
  using T = typename Ar::T;
  constexpr int NW = NT / 32;
  static_assert(NT % 32 == 0 && NW >= 2 && BS_B * BS_B % NT == 0, "at least two warps");
  T* sX = scratch;                                          // [i][l] = X_il, l <= i
  T* red = scratch + BS_B * BS_LD;                          // [warp][r][lane]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nblk = (n + BS_B - 1) / BS_B;
  constexpr int NX = BS_B * BS_B / NT;                      // elements of X per thread
  T xr[NX];
  auto load_x = [&](int k0, int kb) {
#pragma unroll
    for (int q = 0; q < NX; ++q) {
      const int e = threadIdx.x + q * NT, l = e >> 5, i = e & 31;   // consecutive threads: consecutive i
      xr[q] = Ar::zero();
      if (i < kb && l < kb) {
        if (l < i) xr[q] = A[size_t(k0 + l) * n + k0 + i];
        else if (l == i) xr[q] = inv_diag[k0 + i];
      }
    }
  };
  auto store_x = [&]() {
#pragma unroll
    for (int q = 0; q < NX; ++q) {
      const int e = threadIdx.x + q * NT;
      sX[(e & 31) * BS_LD + (e >> 5)] = xr[q];
    }
  };
  {
    // forward: L y = b.  Rows i = warp + NW q of the block; CH column chunks of every row in flight,
    // two sets of them
    constexpr int RPW = (BS_B + NW - 1) / NW, CH = 2;
    T a[2][CH][RPW];
    auto load_a = [&](int k0, int kb, int t0, T (&dst)[CH][RPW]) {
      const int nt = k0 / BS_B;                             // 32-column chunks left of the block
#pragma unroll
      for (int u = 0; u < CH; ++u)
#pragma unroll
        for (int q = 0; q < RPW; ++q) {
          const int i = warp + NW * q;
          dst[u][q] = i < kb && t0 + u < nt ? A[size_t(k0 + i) * n + BS_B * (t0 + u) + lane] : Ar::zero();
        }
    };
    load_x(0, min(BS_B, n));
    for (int bk = 0; bk < nblk; ++bk) {
      const int k0 = bk * BS_B, kb = min(BS_B, n - k0), nt = k0 / BS_B;
      const int k1 = k0 + BS_B, kb1 = min(BS_B, n - k1);
      store_x();
      T s0[RPW], s1[RPW];
#pragma unroll
      for (int q = 0; q < RPW; ++q) { s0[q] = Ar::zero(); s1[q] = Ar::zero(); }
      auto use_a = [&](int t0, const T (&src)[CH][RPW]) {
#pragma unroll
        for (int u = 0; u < CH; ++u) {
          if (t0 + u < nt) {
            const int l = BS_B * (t0 + u) + lane;
            const T y0 = sb[2 * l], y1 = sb[2 * l + 1];
#pragma unroll
            for (int q = 0; q < RPW; ++q) {
              Ar::acc(s0[q], src[u][q], y0);
              Ar::acc(s1[q], src[u][q], y1);
            }
          }
        }
      };
      // sets 0 and 1 (chunks 0 .. 2 CH - 1) were requested during the last block
      for (int t0 = 0; t0 < nt; t0 += 2 * CH) {
        use_a(t0, a[0]);
        if (t0 + 2 * CH < nt) load_a(k0, kb, t0 + 2 * CH, a[0]);
        use_a(t0 + CH, a[1]);
        if (t0 + 3 * CH < nt) load_a(k0, kb, t0 + 3 * CH, a[1]);
      }
      if (bk + 1 < nblk) {
        load_x(k1, kb1);
        load_a(k1, kb1, 0, a[0]);
        load_a(k1, kb1, CH, a[1]);
      }
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const int i = warp + NW * q;
        if (i < kb) {                                         // the same in the whole warp
          const T r0 = Ar::warp_sum(Ar::norm(s0[q])), r1 = Ar::warp_sum(Ar::norm(s1[q]));
          if (lane == 0) {
            sb[2 * (k0 + i)] = Ar::sub(sb[2 * (k0 + i)], r0);
            sb[2 * (k0 + i) + 1] = Ar::sub(sb[2 * (k0 + i) + 1], r1);
          }
        }
      }
      __syncthreads();
      if (warp < 2) {                                         // y_blk = X t
        T y = Ar::zero();
        if (lane < kb)
          for (int l = 0; l <= lane; ++l) Ar::acc(y, sX[lane * BS_LD + l], sb[2 * (k0 + l) + warp]);
        __syncwarp();
        if (lane < kb) sb[2 * (k0 + lane) + warp] = Ar::norm(y);
      }
      __syncthreads();
    }
  }
  {
    // backward: L^T x = y.  U row segments of the block's columns in flight per warp, two sets
    constexpr int U = 8;
    T a[2][U];
    auto load_a = [&](int k0, int kb, int i0, T (&dst)[U]) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        dst[u] = lane < kb && i0 + NW * u < n ? A[size_t(i0 + NW * u) * n + k0 + lane] : Ar::zero();
    };
    auto first = [&](int bk) {                              // a block's first requests
      const int k0 = bk * BS_B, kb = min(BS_B, n - k0), i0 = k0 + kb + warp;
      load_x(k0, kb);
      load_a(k0, kb, i0, a[0]);
      load_a(k0, kb, i0 + NW * U, a[1]);
    };
    first(nblk - 1);
    for (int bk = nblk - 1; bk >= 0; --bk) {
      const int k0 = bk * BS_B, kb = min(BS_B, n - k0);
      store_x();
      T s0 = Ar::zero(), s1 = Ar::zero();
      auto use_a = [&](int i0, const T (&src)[U]) {
        if (lane < kb) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int i = i0 + NW * u;
            if (i < n) {
              Ar::acc(s0, src[u], sb[2 * i]);
              Ar::acc(s1, src[u], sb[2 * i + 1]);
            }
          }
        }
      };
      for (int i0 = k0 + kb + warp; i0 < n; i0 += 2 * U * NW) {
        use_a(i0, a[0]);
        if (i0 + 2 * U * NW < n) load_a(k0, kb, i0 + 2 * U * NW, a[0]);
        use_a(i0 + U * NW, a[1]);
        if (i0 + 3 * U * NW < n) load_a(k0, kb, i0 + 3 * U * NW, a[1]);
      }
      if (bk > 0) first(bk - 1);
      red[(warp * 2) * BS_B + lane] = Ar::norm(s0);
      red[(warp * 2 + 1) * BS_B + lane] = Ar::norm(s1);
      __syncthreads();
      if (warp < 2) {                                         // t, then x_blk = X^T t
        T t = Ar::zero();
        for (int w = 0; w < NW; ++w) t = Ar::add(t, red[(w * 2 + warp) * BS_B + lane]);
        if (lane < kb) sb[2 * (k0 + lane) + warp] = Ar::sub(sb[2 * (k0 + lane) + warp], t);
        __syncwarp();
        T x = Ar::zero();
        if (lane < kb)
          for (int i = lane; i < kb; ++i) Ar::acc(x, sX[i * BS_LD + lane], sb[2 * (k0 + i) + warp]);
        __syncwarp();
        if (lane < kb) sb[2 * (k0 + lane) + warp] = Ar::norm(x);
      }
      __syncthreads();
    }
  }
}

}  // namespace edt
