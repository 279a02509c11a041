// Misfit gradients of the line geometry: J = ||F(c0) V - D||^2 of the Born operator (every
// row; the modelling operator has no evanescent cut) and its gradients with respect to the
// model V(x, z) and to the layer velocities c_l of the reference.
//
// Everything is evaluated in the (p, q) spectral domain.  The data transform D -> D2 is N
// times a unitary map in each of its two lateral axes, so with c_J = 1/N^2
//   J = c_J sum_f sum_{p,q} |R2_f(p, q)|^2,   R2 = s_f sum_j g_p g_q Vhat(p - q) - D2
// (eqs. DMV and M read forward, g_n = g(k_n, z_j; omega~_f), Vhat(k_m, z_j) = sum_x V e^{-i k_m x}).
// Differentiating:
//   dJ/dV(x, z_j)  = 2 c_J Re sum_m Ahat(m, j) e^{+i k_m x},
//                    Ahat(m, j) = sum_{f,p} conj(s_f g_p g_{p-m}) R2(p, p - m)      (adjoint Born)
//   dJ/dg_f(n, j)  = 2 c_J s_f [S1(n, j) + S2(n, j)],
//                    S1(n) = sum_q conj(R2(n, q)) g_q Vhat(n - q),
//                    S2(n) = sum_p conj(R2(p, n)) g_p Vhat(p - n)
//                          = sum_m conj(R2^T(n, n - m)) g_{n-m} conj(Vhat(m))  (V real),
// folded onto the table index |n'| (g depends on k only through k^2), then
//   dJ/dc_l = Re sum_{f,k,j} gbar_f(k, j) dg_f(k, j)/dc_l
// by reverse-mode differentiation of the reflectivity recursion of the depth march, from the
// layer coefficients the march leaves (g itself is recomputed per depth, not stored).
//
// The FP32 table of the mixed path holds sqrt|s_f| g, so s_f g_p g_q = ph_f g32_p g32_q with
// ph_f = s_f/|s_f|, and dJ/dg = sqrt|s_f| dJ/dg32 -> the factor 2 c_J ph_f sqrt|s_f| below.
//
// Kernels per chunk of frequency planes (X holds D2):
//   born_resid     (csrc/born.cu) R2, sum |R2|^2 and the folded planes: one value per class of
//                  entries that share a kernel row product;
//   grad_vhat      (m, j) outputs: Ahat(m) + conj Ahat(-m), m = 0..N/2, accumulated across
//                  frequencies in FP64;
//   grad_gbar      (n, j) outputs on the table index n = 0..N/2: S1 and S2 of both signs;
// then once, in FP64: grad_state (per (f, k, layer): the march's state and the reversed recursions'
// coefficients), grad_field (per
// (f, k, layer): the field's depths of that layer, reversed), grad_reverse (per (f, k): the
// two recursions reversed), grad_layer (the per-layer sums); the inverse lateral DFT of Ahat and a
// finalize kernel.
#include "edt_internal.h"
#include "cplx.cuh"
#include "green_coef.cuh"
#include "warpsum.cuh"

#include <algorithm>

namespace edt {

namespace {

__device__ __forceinline__ int tab_index(int n, int N) { return n <= (N >> 1) ? n : N - n; }

// 1 / b with one real division (the depth march's denominators are O(1e-4 .. 1e1))
__device__ __forceinline__ double2 crcp(double2 b) {
  const double r = 1.0 / (b.x * b.x + b.y * b.y);
  return cmk(b.x * r, -b.y * r);
}

__global__ void grad_zero_kernel(Dev d) {
  const size_t n = size_t(d.N) * d.nz;
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
    d.adj[i] = make_double2(0.0, 0.0);
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i <= d.nlayer; i += blockDim.x) d.gacc[i] = 0.0;
}

// Both contractions below stage their operands in shared memory and keep the sliding legs in
// registers.  A 16-byte shared read costs four cycles of the SM's shared-memory port even when
// it is a broadcast, so a thread has to reuse each coefficient over several depths and each leg
// over several outputs: ZP pairs of depths per lane (64 ZP per CTA) and GN = 8 / ZP outputs per
// thread, 128 multiply-adds per 128 to 160 bytes read.  One depth and eight outputs per thread
// read 144 bytes per 64 multiply-adds and ran at the port's rate: at N = 512, 128 frequencies, 256
// depths, 1.43 ms (vhat) and 2.60 ms (gbar); the whole gradient went from 7.97 to 7.19 ms.
template <int ZP> struct Row {                              // a lane's depths of one table row
  float4 v[ZP];
  __device__ __forceinline__ float2 at(int i) const {
    return i & 1 ? make_float2(v[i >> 1].z, v[i >> 1].w) : make_float2(v[i >> 1].x, v[i >> 1].y);
  }
};
// row r of a shared array of rows of 64 ZP depths: depth pair 32 h + lane
template <int ZP>
__device__ __forceinline__ Row<ZP> row_of(const float2* s, int r, int lane) {
  Row<ZP> o;
  const float4* p = reinterpret_cast<const float4*>(s + size_t(r) * (64 * ZP)) + lane;
#pragma unroll
  for (int h = 0; h < ZP; ++h) o.v[h] = p[32 * h];
  return o;
}
// depth of a lane's element i (two consecutive depths per pair)
__device__ __forceinline__ int lane_z(int i, int lane) { return 64 * (i >> 1) + 2 * lane + (i & 1); }

constexpr int CT = 16;                     // steps per staged chunk

// Chunks are staged one ahead: the next chunk's table rows by asynchronous 16-byte copies into
// slots of the circular buffers that the current chunk does not use, its coefficients through
// registers, while the current one is multiplied (without it the kernels' 16 warps per SM left
// the FP32 pipes idle during the loads, 41 % of their cycles used; one gradient of the 512-point,
// 128-frequency, 256-depth line took 7.17 ms, with it 6.29).
__device__ __forceinline__ void copy16(float2* dst, const float2* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ---- B(m, j) += sum over the classes of m of Re(a) U + Im(a) W ------------------------------
// Every entry (p, q) of the plane appears once: the classes {(p, q), (-q, -p)} of m = p - q and
// their mirror images {(q, p), (-p, -q)} of -m share a = g32_p g32_q, and V = Re sum Ahat(m)
// e^{ikx} needs only B(m) = Ahat(m) + conj Ahat(-m) = conj(a) S + a conj(S'), m = 0..N/2, i.e.
// U = S + conj S', W = -i (S - conj S') with four multiply-adds per class and depth.  For
// m = 2 j or 2 j + 1 the classes are p = t + j (+ 1), q = t - j, t = 0..N/2 (t < N/2 for odd m),
// so the legs of a thread's JT consecutive j slide by one per step of t; the ends t = 0, N/2 of
// even m are their own partners, and m = 0, N/2 their own mirror images.  Consecutive chunks of
// t share all but CT of their rows, which stay where they are (circular buffers).
template <int ZP> struct VhatShape {
  static constexpr int JT = 4 / ZP, VJ = 8 * JT;           // j per thread and per CTA (two m each)
  static constexpr int R = 2 * CT + VJ;                    // rows buffered of either leg
  static constexpr int NC = CT * 2 * VJ;                   // coefficients of a chunk
  static constexpr int SMEM = 2 * R * 64 * ZP * int(sizeof(float2)) + 2 * NC * int(sizeof(float4));
};

template <int ZP>
__global__ void __launch_bounds__(256, 2) grad_vhat_kernel(Dev d, int f0) {
  using S = VhatShape<ZP>;
  constexpr int JT = S::JT, VJ = S::VJ, R = S::R, ZC = 64 * ZP, CQ = S::NC / 256;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* cf = reinterpret_cast<float4*>(smem_raw);        // [2][CT][2 VJ] (U, W) of (t, m)
  float2* gps = reinterpret_cast<float2*>(cf + 2 * S::NC); // row jt + u, u = t + ..., in slot u mod R
  float2* gqs = gps + R * ZC;                              // row u - jt - (VJ - 1), u = t + ..., likewise
  const int N = d.N, H = N / 2, msk = N - 1, nk = d.nk, fi = blockIdx.z, f = f0 + fi;
  const int jt = blockIdx.x * VJ, z0 = blockIdx.y * ZC;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float2* g = d.g32 + size_t(f) * nk * d.nzs + z0;
  const float4* E = d.born_fold + size_t(fi) * 2 * nk * nk;
  const float4* T = E + size_t(nk) * nk;
  const bool live = 2 * (jt + JT * w) <= H;                // the same in the whole warp
  float2 acc[2 * JT][2 * ZP];
#pragma unroll
  for (int k = 0; k < 2 * JT; ++k)
#pragma unroll
    for (int i = 0; i < 2 * ZP; ++i) acc[k][i] = make_float2(0.f, 0.f);
  // rows [lo, hi) of u; depths past nz are not copied (their lanes' sums are not stored)
  auto copy_rows = [&](int lo, int hi) {
    for (int e = threadIdx.x; e < (hi - lo) * (ZC / 2); e += 256) {
      const int u = lo + e / (ZC / 2), zz = 2 * (e % (ZC / 2)), sl = (u % R) * ZC + zz;
      if (z0 + zz >= d.nz) continue;
      copy16(gps + sl, g + size_t(tab_index((jt + u) & msk, N)) * d.nzs + zz);
      copy16(gqs + sl, g + size_t(tab_index((u - VJ + 1 - jt) & msk, N)) * d.nzs + zz);
    }
    copies_commit();
  };
  float4 raw[CQ];                                          // folded values of a chunk, as read
  auto load_coef = [&](int t0) {
#pragma unroll
    for (int i = 0; i < CQ; ++i) {
      const int e = threadIdx.x + 256 * i, mi = e % (2 * VJ);
      const int t = t0 + e / (2 * VJ), m = 2 * jt + mi, odd = m & 1, j = m >> 1;
      raw[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (m <= H && t <= H - odd) {
        int p = t + j + odd, q = t - j;
        if (p > H) p -= N;                                  // signed indices, never both negative
        raw[i] = p >= 0 && q >= 0 ? E[size_t(p) * nk + q]
                                  : T[size_t(p >= 0 ? p : -p) * nk + (q >= 0 ? q : -q)];
      }
    }
  };
  auto store_coef = [&](int t0, float4* dst) {
#pragma unroll
    for (int i = 0; i < CQ; ++i) {
      const int e = threadIdx.x + 256 * i, mi = e % (2 * VJ);
      const int t = t0 + e / (2 * VJ), m = 2 * jt + mi, odd = m & 1;
      float2 S1 = make_float2(raw[i].x, raw[i].y), S2 = make_float2(raw[i].z, raw[i].w);
      if (t + (m >> 1) + odd > H) { const float2 x = S1; S1 = S2; S2 = x; }      // p < 0
      float wt = !odd && (t == 0 || t == H) ? 0.5f : 1.f;
      if (m == 0 || m == H) wt *= 0.5f;
      dst[e] = make_float4(wt * (S1.x + S2.x), wt * (S1.y - S2.y), wt * (S1.y + S2.y), wt * (S2.x - S1.x));
    }
  };
  copy_rows(0, VJ + CT);
  load_coef(0);
  store_coef(0, cf);
  int buf = 0;
  for (int t0 = 0; t0 <= H; t0 += CT, buf ^= 1) {
    copies_wait();
    __syncthreads();                                       // this chunk is staged, the last one done with
    const bool more = t0 + CT <= H;
    if (more) {
      copy_rows(t0 + VJ + CT, t0 + VJ + 2 * CT);
      load_coef(t0 + CT);
    }
    if (live) {
      const float4* cb = cf + buf * S::NC + 2 * JT * w;
      // at t = t0 + tt: P[i] = row p of j = jt + JT w + i (u = t + JT w + i), Q[i] = its row q
      // (u = t + VJ - 1 - JT w - i)
      Row<ZP> P[JT + 1], Q[JT];
#pragma unroll
      for (int i = 0; i <= JT; ++i) P[i] = row_of<ZP>(gps, (t0 + JT * w + i) % R, lane);
#pragma unroll
      for (int i = 0; i < JT; ++i) Q[i] = row_of<ZP>(gqs, (t0 + VJ - 1 - JT * w - i) % R, lane);
      int sp = (t0 + JT * w + JT) % R, sq = (t0 + VJ - 1 - JT * w) % R;
#pragma unroll
      for (int tt = 0; tt < CT; ++tt) {
        if (tt > 0) {
          if (t0 + tt > H) break;
          sp = sp + 1 == R ? 0 : sp + 1;
          sq = sq + 1 == R ? 0 : sq + 1;
#pragma unroll
          for (int i = 0; i < JT; ++i) P[i] = P[i + 1];
          P[JT] = row_of<ZP>(gps, sp, lane);
#pragma unroll
          for (int i = JT - 1; i > 0; --i) Q[i] = Q[i - 1];
          Q[0] = row_of<ZP>(gqs, sq, lane);
        }
#pragma unroll
        for (int i = 0; i < JT; ++i)
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            const float4 c = cb[tt * (2 * VJ) + 2 * i + o];
#pragma unroll
            for (int x = 0; x < 2 * ZP; ++x) {
              const float2 a = P[i + o].at(x) * Q[i].at(x);
              float2& s = acc[2 * i + o][x];
              s.x = fmaf(a.x, c.x, fmaf(a.y, c.z, s.x));
              s.y = fmaf(a.x, c.y, fmaf(a.y, c.w, s.y));
            }
          }
      }
    }
    if (more) store_coef(t0 + CT, cf + (buf ^ 1) * S::NC);
  }
#pragma unroll
  for (int k = 0; k < 2 * JT; ++k) {
    const int m = 2 * (jt + JT * w) + k;
    if (m > H) continue;
#pragma unroll
    for (int x = 0; x < 2 * ZP; ++x) {
      const int z = z0 + lane_z(x, lane);
      if (z >= d.nz) continue;
      double* o = reinterpret_cast<double*>(d.adj + size_t(m) * d.nz + z);
      atomicAdd(o, double(acc[k][x].x));
      atomicAdd(o + 1, double(acc[k][x].y));
    }
  }
}

// ---- gbar_f(n, j), n = 0..N/2 -----------------------------------------------------------------
// The entries whose row a holds g_n are, for every signed q, the class of (n, q) and its mirror
// image: dJ/dg32_n = 2 c_J sum_q g32_q [C1 Re Vhat(n - q) + C2 Im Vhat(n - q)] with
// C1 = conj(S + S'), C2 = i conj(S - S') (the folded values carry conj(s_f)/|s_f|); n = 0 and
// N/2 meet every class twice.  GN consecutive n per thread walking m = n - q: the legs q = n - m
// slide by one per step, Vhat(m) is common to them.  dJ/dc_l sums gbar over near-critical
// wavenumbers with much cancellation, so the FP32 sum over m is taken in two levels (CT terms,
// then the chunks).
template <int ZP> struct GbarShape {
  static constexpr int GN = 8 / ZP, GA = 8 * GN;           // n per thread and per CTA
  static constexpr int R = GA + 2 * CT;                    // rows buffered
  static constexpr int NC = CT * (GA + 1);
  static constexpr int SMEM = (R + 2 * CT) * 64 * ZP * int(sizeof(float2)) + 2 * NC * int(sizeof(float4));
};

template <int ZP>
__global__ void __launch_bounds__(256, 2) grad_gbar_kernel(Dev d, int f0) {
  using S = GbarShape<ZP>;
  constexpr int GN = S::GN, GA = S::GA, R = S::R, ZC = 64 * ZP, CQ = CT * GA / 256;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* cf = reinterpret_cast<float4*>(smem_raw);        // [2][CT][GA + 1] (C1, C2) of (m, n)
  float2* ws = reinterpret_cast<float2*>(cf + 2 * S::NC);  // [2][CT] Vhat rows
  float2* gqs = ws + 2 * CT * ZC;                          // row a0 + GA - 1 - u in slot u mod R
  const int N = d.N, H = N / 2, msk = N - 1, nk = d.nk, fi = blockIdx.z, f = f0 + fi;
  const int a0 = blockIdx.x * GA, z0 = blockIdx.y * ZC;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float2* g = d.g32 + size_t(f) * nk * d.nzs + z0;
  const float2* vh = reinterpret_cast<const float2*>(d.vfull) + z0;     // row m at 2 nz m
  const float4* E = d.born_fold + size_t(fi) * 2 * nk * nk;
  const float4* T = E + size_t(nk) * nk;
  const bool live = a0 + GN * w <= H;                      // the same in the whole warp
  float2 tot[GN][2 * ZP];
#pragma unroll
  for (int k = 0; k < GN; ++k)
#pragma unroll
    for (int i = 0; i < 2 * ZP; ++i) tot[k][i] = make_float2(0.f, 0.f);
  // rows q = n - m: u = GA - 1 - (n - a0) + m; depths past nz are not copied (not stored either)
  auto copy_rows = [&](int lo, int hi, int mc, float2* wb) {
    for (int e = threadIdx.x; e < (hi - lo) * (ZC / 2); e += 256) {
      const int u = lo + e / (ZC / 2), zz = 2 * (e % (ZC / 2));
      if (z0 + zz < d.nz)
        copy16(gqs + (u % R) * ZC + zz, g + size_t(tab_index((a0 + GA - 1 - u) & msk, N)) * d.nzs + zz);
    }
    for (int e = threadIdx.x; e < CT * (ZC / 2); e += 256) {
      const int mi = e / (ZC / 2), zz = 2 * (e % (ZC / 2));
      if (z0 + zz < d.nz) copy16(wb + mi * ZC + zz, vh + size_t(mc + mi) * 2 * d.nz + zz);
    }
    copies_commit();
  };
  float4 raw[CQ];
  auto load_coef = [&](int mc) {
#pragma unroll
    for (int i = 0; i < CQ; ++i) {
      const int e = threadIdx.x + 256 * i, n = a0 + e / CT;
      raw[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (n <= H) {
        int q = (n - mc - e % CT) & msk;
        if (q > H) q -= N;
        raw[i] = q >= 0 ? E[size_t(n) * nk + q] : T[size_t(n) * nk - q];
      }
    }
  };
  auto store_coef = [&](float4* dst) {
#pragma unroll
    for (int i = 0; i < CQ; ++i) {
      const int e = threadIdx.x + 256 * i, al = e / CT, n = a0 + al;
      const float4 c = raw[i];
      const float wt = n == 0 || n == H ? 0.5f : 1.f;
      dst[(e % CT) * (GA + 1) + al] = make_float4(wt * (c.x + c.z), -wt * (c.y + c.w), wt * (c.y - c.w), wt * (c.x - c.z));
    }
  };
  copy_rows(0, GA + CT - 1, 0, ws);
  load_coef(0);
  store_coef(cf);
  int buf = 0;
  for (int mc = 0; mc < N; mc += CT, buf ^= 1) {
    copies_wait();
    __syncthreads();                                       // this chunk is staged, the last one done with
    const bool more = mc + CT < N;
    if (more) {
      copy_rows(mc + GA + CT - 1, mc + GA + 2 * CT - 1, mc + CT, ws + (buf ^ 1) * CT * ZC);
      load_coef(mc + CT);
    }
    if (live) {
      const float4* cb = cf + buf * S::NC + GN * w;
      const float2* wb = ws + buf * CT * ZC;
      // n_k = a0 + GN w + k at m = mc + mi: u = GA - 1 - GN w - k + m
      Row<ZP> win[GN];
      float2 acc[GN][2 * ZP];
#pragma unroll
      for (int k = 0; k < GN; ++k) {
        win[k] = row_of<ZP>(gqs, (mc + GA - 1 - GN * w - k) % R, lane);
#pragma unroll
        for (int i = 0; i < 2 * ZP; ++i) acc[k][i] = make_float2(0.f, 0.f);
      }
      int sq = (mc + GA - 1 - GN * w) % R;
#pragma unroll
      for (int mi = 0; mi < CT; ++mi) {
        if (mi > 0) {
          sq = sq + 1 == R ? 0 : sq + 1;
#pragma unroll
          for (int k = GN - 1; k > 0; --k) win[k] = win[k - 1];
          win[0] = row_of<ZP>(gqs, sq, lane);
        }
        const Row<ZP> v = row_of<ZP>(wb, mi, lane);
#pragma unroll
        for (int k = 0; k < GN; ++k) {
          const float4 c = cb[mi * (GA + 1) + k];
#pragma unroll
          for (int i = 0; i < 2 * ZP; ++i) {
            const float2 vz = v.at(i), gz = win[k].at(i);
            const float tx = fmaf(c.x, vz.x, c.z * vz.y), ty = fmaf(c.y, vz.x, c.w * vz.y);
            acc[k][i].x = fmaf(gz.x, tx, fmaf(-gz.y, ty, acc[k][i].x));
            acc[k][i].y = fmaf(gz.x, ty, fmaf(gz.y, tx, acc[k][i].y));
          }
        }
      }
#pragma unroll
      for (int k = 0; k < GN; ++k)
#pragma unroll
        for (int i = 0; i < 2 * ZP; ++i) tot[k][i] = tot[k][i] + acc[k][i];
    }
    if (more) store_coef(cf + (buf ^ 1) * S::NC);
  }
  // times the scale of Vhat (launch_born_v32)
  const float sc = float(scalbn(2.0 / (double(N) * N) * sqrt(d.fc[f].s_abs), d.born_exp[0]));
  float2* G = d.gbar + size_t(f) * nk * d.nz;
#pragma unroll
  for (int k = 0; k < GN; ++k) {
    const int n = a0 + GN * w + k;
    if (n > H) continue;
#pragma unroll
    for (int i = 0; i < 2 * ZP; ++i) {
      const int z = z0 + lane_z(i, lane);
      if (z < d.nz) G[size_t(n) * d.nz + z] = make_float2(sc * tot[k][i].x, sc * tot[k][i].y);
    }
  }
}

// 128 depths per CTA unless the last 64 of them would all be padding
inline bool wide_depths(int nz) { return (nz + 127) / 128 * 128 - nz < 64; }

cudaError_t vhat_launch(const Dev& d, int f0, int nfc, cudaStream_t s) {
  const int nj = d.N / 4 + 1;                              // m = 0..N/2, two per j
  if (wide_depths(d.nz)) {
    using S = VhatShape<2>;
    grad_vhat_kernel<2><<<dim3((nj + S::VJ - 1) / S::VJ, (d.nz + 127) / 128, nfc), 256, S::SMEM, s>>>(d, f0);
  } else {
    using S = VhatShape<1>;
    grad_vhat_kernel<1><<<dim3((nj + S::VJ - 1) / S::VJ, (d.nz + 63) / 64, nfc), 256, S::SMEM, s>>>(d, f0);
  }
  return cudaGetLastError();
}

cudaError_t gbar_launch(const Dev& d, int f0, int nfc, cudaStream_t s) {
  if (wide_depths(d.nz)) {
    using S = GbarShape<2>;
    grad_gbar_kernel<2><<<dim3((d.nk + S::GA - 1) / S::GA, (d.nz + 127) / 128, nfc), 256, S::SMEM, s>>>(d, f0);
  } else {
    using S = GbarShape<1>;
    grad_gbar_kernel<1><<<dim3((d.nk + S::GA - 1) / S::GA, (d.nz + 63) / 64, nfc), 256, S::SMEM, s>>>(d, f0);
  }
  return cudaGetLastError();
}

// ---- dJ/dc_l: reverse-mode differentiation of the depth march ------------------------------
// Per (f, k), FP64.  Forward: kappa_l, rho_l, r_l, A_l as in the march
// (upward: y = kappa_{l+1}(1 - r_{l+1})/(1 + r_{l+1}), rho_l = (kappa_l - y)/(kappa_l + y),
// r_l = rho_l E_l, E_l = e^{2 i kappa_l h_l}; downward: A_0 = i/(2 kappa_0),
// A_{l+1} = A_l F_l, F_l = e^{i kappa_l h_l}(1 + rho_l)/(1 + r_{l+1}); field
// g(z) = A_l (P + rho_l Q), P = e^{i kappa_l d}, Q = e^{i kappa_l (2 h_l - d)}, d = z - t_l).
// Every step is holomorphic in its inputs, so with dJ = Re(gbar dg) each input's cotangent
// is the sum over its uses of (output cotangent) x (complex partial derivative).  Reverse
// order: the field, the downward recursion (l descending), the upward one (l ascending),
// finally d kappa_l/d c_l = -omega~^2/(c_l^3 kappa_l).
// Reversed, with b(x) the cotangent of x, the two recursions are linear ones along l,
//   b(A_l) += b(A_{l+1}) F_l,
//   b(rho_l) += b(A_{l+1}) P_l + b(r_l) E_l,   b(r_{l+1}) = b(rho_l) X_l - b(A_{l+1}) Q_l,
//   P_l = A_l dF_l/drho_l,  Q_l = -A_l dF_l/dr_{l+1},  X_l = (drho_l/dy)(dy/dr_{l+1}),
// and the kappa_l collect b(A_{l+1}) A_l dF_l/dkappa_l, b(r_l) dr_l/dkappa_l, b(rho_l) U_l and
// b(rho_{l-1}) W_{l-1}, U_l = drho_l/dkappa_l, W_l = (drho_l/dy)(dy/dkappa_{l+1}).  All coefficients
// and collections are formed per layer in parallel; only the recursions themselves, a
// multiply-add or two per layer, run one layer after the other (with everything inside them, two
// reciprocals per layer, they took 0.40 ms for the 512-point line, 128 frequencies and 20 layers).
constexpr int GS_KAP = 0, GS_RHO = 1, GS_A = 2, GS_BKAP = 3, GS_BRHO = 4, GS_BA = 5, GS_F = 6, GS_X = 7, GS_P = 8,
              GS_Q = 9, GS_U = 10, GS_W = 11;
constexpr int GS_BR = GS_X;              // takes X's place as the recursion passes

__device__ __forceinline__ double2& gs_at(const Dev& d, int f, int l, int slot, int k) {
  return d.gscr[((size_t(f) * d.nlayer + l) * GS_SLOTS + slot) * d.nk + k];
}

// kappa_l, rho_l, A_l per (f, k, l) from the depth march's FP64 coefficients (launch_green ran with the
// same reference), and the reversed recursions' coefficients
__global__ void __launch_bounds__(128) grad_state_kernel(Dev d) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int J = d.nlayer;
  if (gid >= (long long)d.nf * J * d.nk) return;
  const int k = int(gid % d.nk);
  const long long fl = gid / d.nk;
  const int l = int(fl % J), f = int(fl / J);
  const GreenLayer q = green_layer_state(d, f, k, l);
  const double2 one = cmk(1.0, 0.0);
  gs_at(d, f, l, GS_KAP, k) = q.kappa;
  gs_at(d, f, l, GS_RHO, k) = q.rho;
  gs_at(d, f, l, GS_A, k) = q.amp;
  if (l == J - 1) return;
  const GreenLayer n = green_layer_state(d, f, k, l + 1);
  const double2 rn = l + 1 < J - 1 ? n.rho * (n.eh * n.eh) : cmk(0.0, 0.0);        // r_{l+1}
  const double2 ir = crcp(one + rn), dy = (one - rn) * ir, y = n.kappa * dy, sm = q.kappa + y, is2 = crcp(sm * sm);
  const double2 P = q.amp * q.eh * ir, up = (one + q.rho) * ir;
  gs_at(d, f, l, GS_F, k) = q.eh * up;
  gs_at(d, f, l, GS_X, k) = (4.0 * q.kappa) * n.kappa * is2 * (ir * ir);
  gs_at(d, f, l, GS_P, k) = P;
  gs_at(d, f, l, GS_Q, k) = P * up;
  gs_at(d, f, l, GS_U, k) = (2.0 * y) * is2;
  gs_at(d, f, l, GS_W, k) = (-2.0 * q.kappa) * is2 * dy;
}

// field, reversed, per (f, k, l): the depths z_j of layer l (a contiguous index range, dz apart)
// give A_l, rho_l, kappa_l their cotangents; gbar on the table index |n'| = k.  With P_i = P_0 E^i,
// E = e^{i kappa dz}, and Q_i = Q_last E^(n-1-i), the four sums over the depths
//   sum gbar P, sum gbar d P, sum gbar Q, sum gbar (2h - d) Q
// are two polynomials in E and their derivatives, evaluated by Horner's rule (|E| <= 1) in 16
// FP64 multiply-adds per depth; the FP64 unit bounds the kernel.  With the coefficients taken from
// the march and these sums, a gradient at 512 points, 128 frequencies, 256 depths and 20 layers takes
// 5.31 ms; with the recursion repeated here and P, Q advanced depth by depth it took 6.29.
// gb64: the cotangent already on the table index in FP64 ([nf][nk][nz]), else d.gbar.
__global__ void __launch_bounds__(128) grad_field_kernel(Dev d, const double2* gb64) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int J = d.nlayer;
  if (gid >= (long long)d.nf * J * d.nk) return;
  const int k = int(gid % d.nk);
  const long long fl = gid / d.nk;
  const int l = int(fl % J), f = int(fl / J);
  // depth range of layer l: first j with z_layer[j] >= l and >= l + 1
  auto lower = [&](int v) {
    int lo = 0, hi = d.nz;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (d.z_layer[mid] < v) lo = mid + 1; else hi = mid;
    }
    return lo;
  };
  const int j0 = lower(l), j1 = lower(l + 1);
  double2 bA = cmk(0.0, 0.0), bRho = bA, bK = bA;
  if (j0 < j1) {
    const double2 kl = gs_at(d, f, l, GS_KAP, k), Al = gs_at(d, f, l, GS_A, k);
    const bool last = l == J - 1;
    const double dz = d.dz;
    const double2 E = cexp(cmk(-kl.y * dz, kl.x * dz));
    const size_t row = (size_t(f) * d.nk + k) * d.nz;
    auto gb = [&](int j) {
      if (gb64) return gb64[row + j];
      const float2 v = d.gbar[row + j];
      return cmk(double(v.x), double(v.y));
    };
    // value and derivative: der = der E + val, val = val E + c
    auto horner = [&](double2& val, double2& der, double2 c) {
      der = cmk(fma(der.x, E.x, fma(-der.y, E.y, val.x)), fma(der.x, E.y, fma(der.y, E.x, val.y)));
      val = cmk(fma(val.x, E.x, fma(-val.y, E.y, c.x)), fma(val.x, E.y, fma(val.y, E.x, c.y)));
    };
    double2 v = cmk(0.0, 0.0), w = v;
    for (int j = j1 - 1; j >= j0; --j) horner(v, w, gb(j));
    const double d0 = d.z_off[j0];
    const double2 P0 = cexp(cmk(-kl.y * d0, kl.x * d0));
    bA = P0 * v;
    double2 s = P0 * (d0 * v + dz * (E * w));                 // sum gbar d P
    if (!last) {
      const double2 rho = gs_at(d, f, l, GS_RHO, k);
      v = w = cmk(0.0, 0.0);
      for (int j = j0; j < j1; ++j) horner(v, w, gb(j));
      const double q = 2.0 * (d.layer_top[l + 1] - d.layer_top[l]) - d.z_off[j1 - 1];   // 2h - d, last depth
      const double2 Q = cexp(cmk(-kl.y * q, kl.x * q));
      const double2 sq = Q * v;
      bA = bA + rho * sq;
      bRho = Al * sq;
      s = s + rho * (Q * (q * v + dz * (E * w)));
    }
    bK = cmk(0.0, 1.0) * (Al * s);
  }
  gs_at(d, f, l, GS_BA, k) = bA;
  gs_at(d, f, l, GS_BRHO, k) = bRho;
  gs_at(d, f, l, GS_BKAP, k) = bK;
}

// the reversed recursions per (f, k), each layer's operands loaded while the one before it is
// worked on
__global__ void __launch_bounds__(32) grad_reverse_kernel(Dev d) {
  const int gid = blockIdx.x * 32 + threadIdx.x, J = d.nlayer;
  if (gid >= d.nf * d.nk) return;
  const int f = gid / d.nk, k = gid - f * d.nk;
  // downward recursion: A_{l+1} = A_l F_l
  double2 bA = gs_at(d, f, J - 1, GS_BA, k);
  double2 F, B;
  auto fetch_a = [&](int l) { F = gs_at(d, f, l, GS_F, k); B = gs_at(d, f, l, GS_BA, k); };
  if (J > 1) fetch_a(J - 2);
  for (int l = J - 2; l >= 0; --l) {
    bA = B + bA * F;
    if (l > 0) fetch_a(l - 1);
    gs_at(d, f, l, GS_BA, k) = bA;
  }
  // upward recursion (l ascending: r_l's cotangent is complete when l is reached)
  double2 bR = cmk(0.0, 0.0), rho, P, Q, X, eh, A1;
  auto fetch_r = [&](int l) {
    rho = gs_at(d, f, l, GS_BRHO, k);
    P = gs_at(d, f, l, GS_P, k);
    Q = gs_at(d, f, l, GS_Q, k);
    X = gs_at(d, f, l, GS_X, k);
    eh = green_layer_eh(d, f, k, l);
    A1 = gs_at(d, f, l + 1, GS_BA, k);
  };
  if (J > 1) fetch_r(0);
  for (int l = 0; l <= J - 2; ++l) {
    const double2 bRho = rho + A1 * P + bR * (eh * eh), next = bRho * X - A1 * Q;
    if (l < J - 2) fetch_r(l + 1);
    gs_at(d, f, l, GS_BRHO, k) = bRho;
    gs_at(d, f, l, GS_BR, k) = bR;
    bR = next;
  }
}

// dJ/dc_l = Re(kappabar_l dkappa_l/dc_l) summed over (f, k): warp sums, one partial per warp and layer
// (added in warp order by the finalize kernel, so the result does not depend on the order the
// warps ran in)
__global__ void __launch_bounds__(128) grad_layer_kernel(Dev d) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x, l = blockIdx.y, f = blockIdx.z;
  const int J = d.nlayer;
  double v = 0.0;
  if (k < d.nk) {
    const double2 kl = gs_at(d, f, l, GS_KAP, k);
    double2 b = gs_at(d, f, l, GS_BKAP, k);
    if (l < J - 1) {
      const double h = d.layer_top[l + 1] - d.layer_top[l];
      const double2 eh = green_layer_eh(d, f, k, l);
      b = b + gs_at(d, f, l + 1, GS_BA, k) * gs_at(d, f, l, GS_A, k) * gs_at(d, f, l, GS_F, k) * cmk(0.0, h);
      b = b + gs_at(d, f, l, GS_BR, k) * gs_at(d, f, l, GS_RHO, k) * (eh * eh) * cmk(0.0, 2.0 * h);
      b = b + gs_at(d, f, l, GS_BRHO, k) * gs_at(d, f, l, GS_U, k);
    }
    if (l > 0) b = b + gs_at(d, f, l - 1, GS_BRHO, k) * gs_at(d, f, l - 1, GS_W, k);
    else b = b + gs_at(d, f, 0, GS_BA, k) * cmk(0.0, -0.5) * crcp(kl * kl);
    const FreqConst fc = d.fc[f];
    const double2 om = cmk(fc.om_re, fc.om_im);
    const double c = d.layer_vel[l];
    v = (b * ((-1.0 / (c * c * c)) * (om * om) * crcp(kl))).x;
  }
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const size_t wid = (size_t(f) * gridDim.x + blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if ((threadIdx.x & 31) == 0) d.gcpart[wid * J + l] = v;
}

// nw: the reverse kernel's warps.  One warp per layer: lane l adds the partials l, l + 32, ... in
// order, then a butterfly over the lanes (a fixed order of additions).
__global__ void __launch_bounds__(32) grad_finalize_kernel(Dev d, double* J, double* gc, int nw) {
  const int l = blockIdx.x, lane = threadIdx.x;
  if (l == 0 && lane == 0 && J) J[0] = d.gacc[0] / (double(d.N) * d.N);
  double t = 0.0;
  for (int w = lane; w < nw; w += 32) t += d.gcpart[size_t(w) * d.nlayer + l];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) gc[l] = t;
}

// ---- adjoint of the inversion D -> V (linear in D: G and lam depend on the rows only) --------
// V = (1/N) Re sum_m Vhat(m) e^{i k_m x} with Vhat(m) = x_+ + i x_- for m = 0..N/2 and the
// conjugate for -m, so dV/dx_+(m) = (c_m/N) cos(k_m x), dV/dx_-(m) = -(c_m/N) sin(k_m x),
// c_m = 1 at the self-paired m (x_- = 0 there) and 2 otherwise: xbar(m) = (c_m/N) DFT(Vbar)(m).
// xbar goes where the forward solve reads b.
__global__ void adj_xbar_kernel(Dev d) {
  const int m = blockIdx.x, N = d.N;
  const bool self = m == 0 || 2 * m == N;
  const double c = (self ? 1.0 : 2.0) / double(N);
  for (int z = threadIdx.x; z < d.nz; z += blockDim.x) {
    const double2 v = d.vfull[size_t(m) * d.nz + z];
    d.b[(size_t(m) * d.nz + z) * 2 + 0] = c * v.x;
    d.b[(size_t(m) * d.nz + z) * 2 + 1] = self ? 0.0 : c * v.y;
  }
}

// r += xbar: with zero right-hand sides the refinement kernel leaves r = -Ahat^T Ahat y, so
// this makes r - lam y = xbar - (Ahat^T Ahat + lam I) y, the residual of the adjoint solve.
__global__ void adj_addb_kernel(Dev d) {
  const size_t n = size_t(d.nsub) * d.nz * 2;
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
    d.r[i] += d.b[i];
}

// table rows |p|, |q| of a row of subproblem m
__device__ __forceinline__ int2 table_rows(const Dev& d, int m, uint32_t row) {
  const int p = row_p(row), q = (p - m) & (d.N - 1), t0 = row_f(row) * d.nk;
  return make_int2(t0 + tab_index(p, d.N), t0 + tab_index(q, d.N));
}

// Products of two rows a = g32_p g32_q, whose table rows lanes i0 and i1 hold in tr, with two depth
// vectors va, vb, lanes over depth: lane 16 h + 4 c returns row h's sum (a.va re, im, a.vb re, im)_c.
__device__ __forceinline__ float row_pair_dots(const Dev& d, int2 tr, int i0, int i1, const float* va, const float* vb,
                                               int lane) {
  const float2* g[2][2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    g[h][0] = d.g32 + size_t(__shfl_sync(0xffffffffu, tr.x, h ? i1 : i0)) * d.nzs;
    g[h][1] = d.g32 + size_t(__shfl_sync(0xffffffffu, tr.y, h ? i1 : i0)) * d.nzs;
  }
  float s[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) s[c] = 0.f;
#pragma unroll 4
  for (int z = lane; z < d.nz; z += 32) {
    const float a = va[z], b = vb[z];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 t = g[h][0][z] * g[h][1][z];
      s[4 * h + 0] = fmaf(t.x, a, s[4 * h + 0]); s[4 * h + 1] = fmaf(t.y, a, s[4 * h + 1]);
      s[4 * h + 2] = fmaf(t.x, b, s[4 * h + 2]); s[4 * h + 3] = fmaf(t.y, b, s[4 * h + 3]);
    }
  }
  return warp_sums(s, lane);
}

// Per kept row (f, p) of m at frequencies [f0, f1), with bbar = (G + lam I)^-1 xbar in d.x:
// b_+- = sum_rows w Re(conj(row) rhs_+-) gives rhsbar = w sum_z row(z) bbar(z); then the
// rotation rhs = rot d, the split d_+ = (a + c)/2, d_- = (a - c)/(2i) with a = D2(p, q),
// c = D2(q, p) (folded rows: a and c the means with D2(-q, -p), D2(-p, -q)) are reversed and
// scattered (atomically) into the chunk's planes X[fi][q][p] = D2bar(p, q).
__global__ void __launch_bounds__(256) adj_rows_kernel(Dev d, int f0, int f1) {
  __shared__ float bb[2][512];                        // bbar_+, bbar_- per depth, nz <= 512
  const int m = blockIdx.y, N = d.N, msk = N - 1;
  if (d.status[m] != EDT_OK) return;
  const double* yb = d.x + size_t(m) * d.nz * 2;
  for (int z = threadIdx.x; z < d.nz; z += blockDim.x) {
    bb[0][z] = float(yb[2 * z]);
    bb[1][z] = float(yb[2 * z + 1]);
  }
  __syncthreads();
  const long long r0 = d.row_off_mf[size_t(m) * (d.nf + 1) + f0];
  const long long r1 = d.row_off_mf[size_t(m) * (d.nf + 1) + f1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  float2* X = reinterpret_cast<float2*>(d.X);
  // two rows per warp, lanes over depth; lane 16 h ends with row h's sums
  const long long step = 2LL * gridDim.x * nwarp;
  for (long long rb = r0 + 2 * ((long long)blockIdx.x * nwarp + warp); rb < r1; rb += step) {
    const bool two = rb + 1 < r1;
    const long long ri = rb + (two ? lane >> 4 : 0);
    const uint32_t row = d.rows[ri];
    const int f = row_f(row), p = row_p(row), q = (p - m) & msk;
    const int2 tr = table_rows(d, m, row);
    const float s = row_pair_dots(d, tr, 0, 16, bb[0], bb[1], lane);
    const int l0 = lane & 16;
    const float2 sp = make_float2(__shfl_sync(0xffffffffu, s, l0), __shfl_sync(0xffffffffu, s, l0 + 4));
    const float2 sm = make_float2(__shfl_sync(0xffffffffu, s, l0 + 8), __shfl_sync(0xffffffffu, s, l0 + 12));
    if (lane != 0 && !(lane == 16 && two)) continue;
    const bool w2 = row_w2(row);
    const FreqConst fc = d.fc[f];
    const float2 crot = make_float2(float(fc.rot_re), float(-fc.rot_im));   // conj(rot)
    const float w = w2 ? 2.f : 1.f;
    const float2 dp = crot * (w * sp), dm = crot * (w * sm);
    // abar = dp/2 + (i/2) dm, cbar = dp/2 - (i/2) dm; folded rows split each in halves
    const float h = w2 ? 0.25f : 0.5f;
    const float2 abar = make_float2(h * (dp.x - dm.y), h * (dp.y + dm.x));
    const float2 cbar = make_float2(h * (dp.x + dm.y), h * (dp.y - dm.x));
    float2* P = X + size_t(f - f0) * N * N;
    auto add = [&](int pp, int qq, float2 v) {             // D2bar(pp, qq) at X[qq][pp]
      float* o = reinterpret_cast<float*>(P + size_t(qq & msk) * N + (pp & msk));
      atomicAdd(o, v.x);
      atomicAdd(o + 1, v.y);
    };
    add(p, q, abar);
    add(q, p, cbar);
    if (w2) {
      add(-q, -p, abar);
      add(-p, -q, cbar);
    }
  }
}

// ---- dL/dc_l through the damped solve ----------------------------------------------------
// Per subproblem m, x solves (Ahat^T Ahat + lam I) x = Ahat^T dhat with lam = alpha tr(Ahat^T
// Ahat) (the Gram's trace, the sum of w |A|^2 over the rows); the kernel rows A = g32_p g32_q
// (g32 = sqrt|s_f| g; the data carry the unit phase of s_f) depend on the reference.  With
// mu = (Ahat^T Ahat + lam I)^-1 xbar, differentiating the normal equations gives the
// cotangent of a complex row (dL = Re sum_z conj(Abar) dA)
//   Abar = w [ sum_k (u_k mu_k + v_k x_k) + gamma A ],
//   u_k = d_k - A . x_k,  v_k = -A . mu_k,  gamma = -2 alpha sum_k mu_k . x_k,
// (k over the two right-hand sides +-; w = 2 for a folded row).  With dA = sqrt|s_f| (g32_q dg_p
// + g32_p dg_q) the table's cotangent in the convention dL = Re sum gbar dg is
//   gbar(f, |p|) += sqrt|s_f| g32_q conj(Abar),   gbar(f, |q|) += sqrt|s_f| g32_p conj(Abar),
// gathered per table row over the rows that read it (row groups built with the plan, in row
// order: no atomics), FP32 products, FP64 sums; then the depth march is reversed as for the
// misfit gradient.
constexpr int IG_WARPS = 8, IG_RPW = 16;             // 128 rows per CTA of the row products

// Per row the products with the depth vectors of its subproblem: mode 0 (before the adjoint
// solve) u_k = d_k - A . x_k with x the forward solution (Vhat), mode 1 v_k = -A . mu_k with mu
// in x; the first CTA of each subproblem also stores the FP32 vectors and, in mode 1, gamma.
__global__ void __launch_bounds__(IG_WARPS * 32) ig_rowdot_kernel(Dev d, int mode) {
  __shared__ float vs[2][512];
  __shared__ double red[IG_WARPS];
  const int m = blockIdx.y, nz = d.nz;
  const bool ok = d.status[m] == EDT_OK;
  const long long r0 = d.row_off[m], nr = d.row_off[m + 1] - r0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double bsum = 0.0;
  for (int z = threadIdx.x; z < nz; z += blockDim.x) {
    float a = 0.f, b = 0.f;
    if (ok) {
      if (mode) {
        const double mp = d.x[(size_t(m) * nz + z) * 2], mm = d.x[(size_t(m) * nz + z) * 2 + 1];
        const double2 xv = d.vhat[size_t(m) * nz + z];
        bsum += mp * xv.x + mm * xv.y;
        a = float(mp); b = float(mm);
      } else {
        const double2 xv = d.vhat[size_t(m) * nz + z];
        a = float(xv.x); b = float(xv.y);
      }
    }
    vs[0][z] = a; vs[1][z] = b;
    if (blockIdx.x == 0) {
      float4* o = d.xmu + size_t(m) * nz + z;
      if (mode) { o->z = a; o->w = b; } else { o->x = a; o->y = b; }
    }
  }
  if (mode && blockIdx.x == 0) {
    for (int o = 16; o > 0; o >>= 1) bsum += __shfl_xor_sync(0xffffffffu, bsum, o);
    if (lane == 0) red[warp] = bsum;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < IG_WARPS; ++w) t += red[w];
      d.gam[m] = ok ? -2.0 * d.alpha * t : 0.0;
    }
  }
  __syncthreads();
  const long long wb = (long long)blockIdx.x * IG_WARPS * IG_RPW + warp * IG_RPW;
  const long long we = min(nr, wb + IG_RPW);
  const int cnt = int(max(0LL, we - wb));
  const float* rhs = reinterpret_cast<const float*>(d.rhs);    // [row][+ re, + im, - re, - im]
  // lane i holds row i's table rows, so that a pair's loads wait for no metadata
  const int2 tr = lane < cnt ? table_rows(d, m, d.rows[r0 + wb + lane]) : make_int2(0, 0);
  for (int i = 0; i < cnt; i += 2) {
    const float s = row_pair_dots(d, tr, i, min(i + 1, cnt - 1), vs[0], vs[1], lane);
    const int c = lane >> 2, row = i + (c >> 2);
    if ((lane & 3) == 0 && row < cnt) {
      const size_t at = size_t(r0 + wb + row);
      float* o = reinterpret_cast<float*>(d.rowc + 2 * at + mode) + (c & 3);
      *o = !ok ? 0.f : mode ? -s : rhs[4 * at + (c & 3)] - s;
    }
  }
}

// One warp per table row (f, n), n = 0 .. N/2, and 32 NZL depths, lanes over depth (NZL per lane): gbar of that
// row from every row that reads it, in row order; 32 rows summed in FP32, then into FP64.  Lane l
// reads the metadata of the 32 rows' l-th and hands it round by shuffles, so the depth loads of
// successive rows wait for nothing but their turn (each row's chain of three dependent loads
// before its depths made the kernel 21 % of an inversion with its vector-Jacobian products).  More than
// 128 depths go to several warps: eight depths per lane left 16 warps per SM (dL/dc of the 512-point
// line with 256 depths 4.70 ms, 4.03 with four).
template <int NZL>
__global__ void __launch_bounds__(256) ig_gather_kernel(Dev d) {
  const long long te = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (te >= (long long)d.nf * d.nk) return;
  const int lane = threadIdx.x & 31, nz = d.nz, N = d.N, msk = N - 1, z0 = 32 * NZL * blockIdx.y + lane;
  const int f = int(te / d.nk);
  const float2* gs = d.g32 + size_t(te) * d.nzs;
  float2 self[NZL], part[NZL];
  double2 acc[NZL];
#pragma unroll
  for (int t = 0; t < NZL; ++t) {
    const int z = z0 + 32 * t;
    self[t] = z < nz ? gs[z] : make_float2(0.f, 0.f);
    part[t] = make_float2(0.f, 0.f);
    acc[t] = make_double2(0.0, 0.0);
  }
  const long long b0 = d.tref_off[te], b1 = d.tref_off[te + 1];
  for (long long base = b0; base < b1; base += 32) {
    const int cnt = int(min(32LL, b1 - base));
    int li = 0, lg = 0, lm = 0;                          // row, other table row, m (w2 in the sign)
    float lgam = 0.f;
    if (lane < cnt) {
      const int2 rf = d.tref[base + lane];
      const uint32_t row = d.rows[rf.x];
      const int m = rf.y >> 1, p = row_p(row), q = (p - m) & msk;
      li = rf.x;
      lg = f * d.nk + tab_index(rf.y & 1 ? p : q, N);
      lm = row_w2(row) ? ~m : m;
      lgam = float(d.gam[m]);
    }
#pragma unroll 2
    for (int k = 0; k < cnt; ++k) {
      const int ri = __shfl_sync(0xffffffffu, li, k), mw = __shfl_sync(0xffffffffu, lm, k);
      const float2* go = d.g32 + size_t(__shfl_sync(0xffffffffu, lg, k)) * d.nzs;
      const float gam = __shfl_sync(0xffffffffu, lgam, k);
      const float4 u = d.rowc[2 * size_t(ri)], v = d.rowc[2 * size_t(ri) + 1];
      const float w = mw < 0 ? 2.f : 1.f;
      const float4* xm = d.xmu + size_t(mw < 0 ? ~mw : mw) * nz;
#pragma unroll
      for (int t = 0; t < NZL; ++t) {
        const int z = z0 + 32 * t;
        if (z < nz) {
          const float2 g2 = go[z];
          const float4 xv = xm[z];                       // (x_+, x_-, mu_+, mu_-)
          const float2 A = self[t] * g2;
          float2 ab;
          ab.x = fmaf(u.x, xv.z, fmaf(u.z, xv.w, fmaf(v.x, xv.x, fmaf(v.z, xv.y, gam * A.x))));
          ab.y = fmaf(u.y, xv.z, fmaf(u.w, xv.w, fmaf(v.y, xv.x, fmaf(v.w, xv.y, gam * A.y))));
          ab.x *= w; ab.y *= w;
          part[t].x = fmaf(g2.x, ab.x, fmaf(g2.y, ab.y, part[t].x));      // g2 conj(ab)
          part[t].y = fmaf(g2.y, ab.x, fmaf(-g2.x, ab.y, part[t].y));
        }
      }
    }
    if (cnt == 32) {
#pragma unroll
      for (int t = 0; t < NZL; ++t) {
        acc[t].x += double(part[t].x); acc[t].y += double(part[t].y);
        part[t] = make_float2(0.f, 0.f);
      }
    }
  }
  const double sq = sqrt(d.fc[f].s_abs);
  double2* out = d.g64 + size_t(te) * nz;
#pragma unroll
  for (int t = 0; t < NZL; ++t) {
    const int z = z0 + 32 * t;
    if (z < nz) out[z] = make_double2(sq * (acc[t].x + double(part[t].x)), sq * (acc[t].y + double(part[t].y)));
  }
}

}  // namespace

// The forward solve with k refinement steps is x = sum_{i<=k} (I - Ht^-1 H)^i Ht^-1 b (Ht the
// factored matrix, H = Ahat^T Ahat + lam I from the rows), a symmetric map: its transpose is
// the same iteration applied to xbar, run here with the forward's own kernels.
cudaError_t launch_invert_vjp(const Dev& d0, const void* Vbar, int Vbar_dtype, void* Dbar, int Dbar_dtype,
                              double* gc, int refine, cudaStream_t s) {
  cudaError_t e;
  // the adjoint solve's refinement residual is xbar - (Ahat^T Ahat + lam I) y: the rows'
  // data term is left out (the right-hand sides stay for later calls)
  Dev d = d0;
  d.refine_nodata = 1;
  const dim3 rg(unsigned((std::max(d.rows_max_sub, 1LL) + IG_WARPS * IG_RPW - 1) / (IG_WARPS * IG_RPW)), d.nsub);
  if (gc) {
    ig_rowdot_kernel<<<rg, IG_WARPS * 32, 0, s>>>(d, 0);          // u = d - A x
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if ((e = launch_lateral_dft(d, Vbar, Vbar_dtype, s)) != cudaSuccess) return e;
  adj_xbar_kernel<<<d.nsub, 256, 0, s>>>(d);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_chol_resolve(d, s)) != cudaSuccess) return e;
  for (int it = 0; it < refine; ++it) {
    if ((e = launch_refine(d, s)) != cudaSuccess) return e;
    adj_addb_kernel<<<152, 256, 0, s>>>(d);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_refine_update(d, s)) != cudaSuccess) return e;
  }
  if (Dbar) {
    for (int f0 = 0; f0 < d.nf; f0 += d.fchunk) {
      const int nfc = std::min(d.fchunk, d.nf - f0);
      if ((e = cudaMemsetAsync(d.X, 0, size_t(nfc) * d.N * d.N * sizeof(float2), s)) != cudaSuccess) return e;
      adj_rows_kernel<<<dim3(32, d.nsub), 256, 0, s>>>(d, f0, f0 + nfc);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      if ((e = launch_transform_adjoint(d, Dbar, Dbar_dtype, f0, nfc, s)) != cudaSuccess) return e;
    }
  }
  if (gc) {
    ig_rowdot_kernel<<<rg, IG_WARPS * 32, 0, s>>>(d, 1);          // v = -A mu, gamma
    const unsigned gg = unsigned(((long long)d.nf * d.nk + 7) / 8);
    if (d.nz <= 64) ig_gather_kernel<2><<<gg, 256, 0, s>>>(d);
    else ig_gather_kernel<4><<<dim3(gg, (d.nz + 127) / 128), 256, 0, s>>>(d);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    grad_zero_kernel<<<152, 256, 0, s>>>(d);
    // the forward solve's depth march may have been the FP32 one: its FP64 coefficients
    if ((e = launch_green(d, s, GREEN_COEF)) != cudaSuccess) return e;
    const dim3 gk((d.nk + 127) / 128, d.nf);
    const long long nfl = (long long)d.nf * d.nlayer * d.nk;
    grad_state_kernel<<<unsigned((nfl + 127) / 128), 128, 0, s>>>(d);
    grad_field_kernel<<<unsigned((nfl + 127) / 128), 128, 0, s>>>(d, d.g64);
    grad_reverse_kernel<<<unsigned((d.nf * d.nk + 31) / 32), 32, 0, s>>>(d);
    grad_layer_kernel<<<dim3(gk.x, d.nlayer, d.nf), 128, 0, s>>>(d);
    grad_finalize_kernel<<<d.nlayer, 32, 0, s>>>(d, nullptr, gc, int(gk.x * gk.y * 4));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t prepare_grad() {
  cudaError_t e;
  if ((e = allow_smem(grad_vhat_kernel<1>, VhatShape<1>::SMEM)) != cudaSuccess) return e;
  if ((e = allow_smem(grad_vhat_kernel<2>, VhatShape<2>::SMEM)) != cudaSuccess) return e;
  if ((e = allow_smem(grad_gbar_kernel<1>, GbarShape<1>::SMEM)) != cudaSuccess) return e;
  return allow_smem(grad_gbar_kernel<2>, GbarShape<2>::SMEM);
}

bool grad_supported(const Dev& d) {
  return d.geom == EDT_GEOM_LINE && d.precision == EDT_MIXED && d.N >= 64 && d.nlayer <= GRAD_MAX_LAYERS &&
         d.gscr != nullptr;
}

// Adjoint Born operator of the line geometry, V = F^T D for <D1, D2> = Re sum conj(D1) D2 and
// <V1, V2> = sum V1 V2: the adjoint of the inverse data transform is T / N^2 (T the data
// transform, N times a unitary map per axis), then Vbar_hat(m, z) = sum_f sum_p
// conj(s_f g(k_p, z) g(k_{p-m}, z)) D2(p, p - m) and V(x, z) = Re sum_m Vbar_hat(m, z) e^{+i k_m x}.
// Mixed path: FP32 transform and the misfit gradient's adjoint-Born contraction (FP64 sums
// across frequencies); FP64 path: FP64 transform and a direct FP64 contraction.
cudaError_t launch_adjoint(const Dev& d, const void* D, int D_dtype, void* V, int V_dtype, cudaStream_t s) {
  cudaError_t e;
  const int N = d.N;
  const double scale = 1.0 / (double(N) * N);
  if (d.precision == EDT_FP64) {
    if ((e = cudaMemsetAsync(d.vfull, 0, sizeof(double2) * size_t(N) * d.nz, s)) != cudaSuccess) return e;
    for (int f0 = 0; f0 < d.nf; f0 += d.fchunk) {
      const int nfc = std::min(d.fchunk, d.nf - f0);
      if ((e = launch_adjoint64_chunk(d, D, D_dtype, f0, nfc, s)) != cudaSuccess) return e;
    }
    return launch_lateral_idft_real(d, d.vfull, scale, V, V_dtype, s);
  }
  grad_zero_kernel<<<152, 256, 0, s>>>(d);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  for (int f0 = 0; f0 < d.nf; f0 += d.fchunk) {
    const int nfc = std::min(d.fchunk, d.nf - f0);
    if ((e = launch_transform<float>(d, D, D_dtype, f0, nfc, s)) != cudaSuccess) return e;
    if ((e = launch_born_residual(d, f0, nfc, false, s)) != cudaSuccess) return e;
    if ((e = vhat_launch(d, f0, nfc, s)) != cudaSuccess) return e;
  }
  return launch_lateral_idft_real(d, d.adj, scale, V, V_dtype, s);
}

cudaError_t launch_misfit_grad(const Dev& d, const void* V, int V_dtype, const void* D, int D_dtype,
                               double* J, void* gV, double* gc, cudaStream_t s) {
  cudaError_t e;
  grad_zero_kernel<<<152, 256, 0, s>>>(d);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_lateral_dft(d, V, V_dtype, s, born_v32_exps(d))) != cudaSuccess) return e;
  if ((e = launch_born_v32(d, s)) != cudaSuccess) return e;
  const int N = d.N;
  for (int f0 = 0; f0 < d.nf; f0 += d.fchunk) {
    const int nfc = std::min(d.fchunk, d.nf - f0);
    if ((e = launch_transform<float>(d, D, D_dtype, f0, nfc, s)) != cudaSuccess) return e;
    if ((e = launch_born_residual(d, f0, nfc, true, s)) != cudaSuccess) return e;
    if ((e = vhat_launch(d, f0, nfc, s)) != cudaSuccess) return e;
    if ((e = gbar_launch(d, f0, nfc, s)) != cudaSuccess) return e;
  }
  const dim3 gk((d.nk + 127) / 128, d.nf);
  const long long nfl = (long long)d.nf * d.nlayer * d.nk;
  grad_state_kernel<<<unsigned((nfl + 127) / 128), 128, 0, s>>>(d);
  grad_field_kernel<<<unsigned((nfl + 127) / 128), 128, 0, s>>>(d, nullptr);
  grad_reverse_kernel<<<unsigned((d.nf * d.nk + 31) / 32), 32, 0, s>>>(d);
  grad_layer_kernel<<<dim3(gk.x, d.nlayer, d.nf), 128, 0, s>>>(d);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_lateral_idft_real(d, d.adj, 2.0 / (double(N) * N), gV, V_dtype, s)) != cudaSuccess) return e;
  grad_finalize_kernel<<<d.nlayer, 32, 0, s>>>(d, J, gc, int(gk.x * gk.y * 4));
  return cudaGetLastError();
}

}  // namespace edt
